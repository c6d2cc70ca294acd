// Fermionic observables (Sec. 5.2): Majorana bilinears on the physical modes
// for every chain, from the inverses W_nm = M_nm(G)^{-1} the sampler keeps.
//
// Contracting the virtual modes of the site states with the bond operator
// X_nm leaves a Gaussian operator on the physical Majoranas whose covariance
// is the Schur complement
//   Gamma_eff^nm = A + B W_nm B^T,
// A the sites' physical blocks and B their physical-virtual couplings (both
// block diagonal by site; the twist sits on the bond side of M = D + O Gamma_X
// O^T, so A and B are untwisted).  By Wick's theorem
//   <psi_n(G)| c_a c_b |psi_m(G)> = N_nm(G) (-i Gamma_eff^nm[a, b])   (a != b).
// Entry (a on site s, b on site t) needs only the B x B block W[site s, site t].
// A and B are real and M_mn = conj(M_nm), so Gamma_eff^mn = A + conj(B W_nm B^T):
// one product serves both orders of a pair n < m.  Outputs per chain:
//   site[s]           = sum_nm lambda_n^* lambda_m <psi_n|c_2s c_2s+1|psi_m> / N(G)
//   link[l][alpha][beta] = same for c_{2s+alpha} c_{2t+beta}, link l = (s -> t)
// (densities n_s = (1 + i site[s]) / 2; hoppings and pairings are linear in
// the link block, and link_term_kernel forms the gauge-invariant one with the
// link operator, u_l F_s F_t, from it).
//
// What bounds it: the latency of the block loads; 32 chains of 8 x 8 U(1), K = 2:
// bilinears 155 us with one thread per item, 60 with a group of B lanes
// (one row of the block each); the four-point function 329 and 89.  Where the
// chains fill the chip, the FP64 unit: 1024 chains of 8 x 8 Z2 178 -> 114 and
// 188 -> 165 us.
#include "ggf_obs_group.cuh"

namespace {

constexpr int FTHREADS = 128;

// A group of BW lanes per (chain, item): items 0 .. V - 1 are sites, the
// others links.
template <class RW, class CW, int BW>
__global__ void __launch_bounds__(OT) fermion_kernel(DevConst dc, int blocks_per_chain, int it0, int items, const RW* Wr,
                                                     const CW* Wc, const cxd* ell, const cxd* ready, cxd* site_out, cxd* link_out,
                                                     cxd* pair_site, cxd* pair_link) {
    constexpr int NG = OT / BW;
    __shared__ PairWeights pw;
    const Geometry& g = dc.g;
    const int c = blockIdx.x / blocks_per_chain, lane = threadIdx.x % BW, K = dc.K;
    const int want = (blockIdx.x - c * blocks_per_chain) * NG + threadIdx.x / BW;
    const bool live = want < items;
    const int it = it0 + min(want, items - 1);
    chain_weights(dc, c, ell, ready, pw);
    const FermionLane f = fermion_lane<BW>(g, K, c, it, lane);
    cxd* out = f.is_site ? site_out : link_out;
    cxd* pout = f.is_site ? pair_site : pair_link;
    cxd* q = pout && live && f.entry ? pout + f.pair : nullptr;
    const size_t NN = (size_t)g.N * g.N;
    cxd acc = {0.0, 0.0};
    for (int p = 0; p < dc.P; ++p) {
        if (p >= K) {
            const cxd x = coupled_entry<CW, BW>(dc, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, f.s, f.t, lane);
            fermion_term(dc, f, p, pw.np[p], pw.E[p], x, acc, q);
        } else {
            const double x = coupled_entry<RW, BW>(dc, Wr + ((size_t)c * K + p) * NN, f.s, f.t, lane);
            fermion_term(dc, f, p, pw.np[p], pw.E[p], x, acc, q);
        }
    }
    // -i (A + sum_p weight_p X_p); A enters with the total weight
    // sum_nm lambda_n^* lambda_m N_nm / N(G) = 1 (only where s == t)
    if (out && live && f.entry) out[f.out] = pair_bilinear(dc, f.s, f.t, f.a, f.b, acc);
}

// A group of BW lanes per (chain, link).
template <class RW, class CW, int BW>
__global__ void __launch_bounds__(OT) fermion4_kernel(DevConst dc, int blocks_per_chain, const RW* Wr, const CW* Wc,
                                                      const cxd* ell, const cxd* ready, cxd* out, cxd* pair_out) {
    constexpr int NG = OT / BW;
    __shared__ PairWeights pw;
    const Geometry& g = dc.g;
    const int c = blockIdx.x / blocks_per_chain, lane = threadIdx.x % BW, K = dc.K;
    const int want = (blockIdx.x - c * blocks_per_chain) * NG + threadIdx.x / BW;
    const bool live = want < g.n_links;
    const int l = min(want, g.n_links - 1);
    chain_weights(dc, c, ell, ready, pw);
    int a0, b0;
    link_ends(g, l, a0, b0);
    const int s = a0 / g.B, t = b0 / g.B;
    cxd* q = pair_out ? pair_out + ((size_t)c * g.n_links + l) * K * K : nullptr;
    const size_t NN = (size_t)g.N * g.N;
    cxd acc = {0.0, 0.0};
    for (int p = 0; p < dc.P; ++p) {
        cxd* po = live ? q : nullptr;
        if (p >= K) {
            cxd g01, g23, x[4];
            four_point_blocks<CW, BW>(dc, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, s, t, lane, g01, g23, x);
            four_point_term(dc, p, lane, s, t, g01, g23, x, pw.np[p], pw.E[p], acc, po);
        } else {
            double g01, g23, x[4];
            four_point_blocks<RW, BW>(dc, Wr + ((size_t)c * K + p) * NN, s, t, lane, g01, g23, x);
            four_point_term(dc, p, lane, s, t, g01, g23, x, pw.np[p], pw.E[p], acc, po);
        }
    }
    acc = acc + shfl_xor_(acc, 1);
    if (out && live && lane == 0) out[(size_t)c * g.n_links + l] = s == t ? cxd{-1.0, 0.0} : acc;
}

// One thread per (chain, link).
__global__ void __launch_bounds__(FTHREADS) link_term_kernel(DevConst dc, int n_chains, const void* links,
                                                             const int* q, const cxd* blk, const cxd* pair_blk,
                                                             cxd* out, cxd* pair_out) {
    const long long t = (long long)blockIdx.x * FTHREADS + threadIdx.x;
    if (t >= (long long)n_chains * dc.g.n_links) return;
    const int c = (int)(t / dc.g.n_links), l = (int)(t - (long long)c * dc.g.n_links);
    link_term_item(dc, c, l, links, q, blk, pair_blk, out, pair_out);
}

}  // namespace

ggf_status ggf_flush(ggf_ctx* ctx, cudaStream_t st);
ggf_status ggf_fermion(ggf_ctx* ctx, cxd* d_site, cxd* d_link, cxd* d_pair_site, cxd* d_pair_link,
                       cudaStream_t st);

// Gauge-invariant link terms of every chain into d_out [n][n_links] and/or
// their per-pair parts into d_pair_out [n][n_links][K][K] (device; either may
// be null), through the link blocks written to the scratch buffers d_blk
// [n][n_links][2][2] and d_pair_blk [n][n_links][2][2][K][K]; d_q [V] device.
ggf_status ggf_link_terms(ggf_ctx* ctx, const int* d_q, cxd* d_blk, cxd* d_pair_blk, cxd* d_out, cxd* d_pair_out,
                          cudaStream_t st) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    if (!d_out) d_blk = nullptr;
    if (!d_pair_out) d_pair_blk = nullptr;
    if (!d_blk && !d_pair_blk) return GGF_OK;
    GGF_TRY(ggf_fermion(ctx, nullptr, d_blk, nullptr, d_pair_blk, st));
    const long long items = (long long)ch.n * g.n_links;
    const long long blocks = (items + FTHREADS - 1) / FTHREADS;
    if (blocks > 0x7fffffffLL) return ggf_fail(ctx, GGF_EINVAL, "too many chains for one launch");
    link_term_kernel<<<(unsigned)blocks, FTHREADS, 0, st>>>(ctx->dc(), ch.n, ch.links, d_q, d_blk, d_pair_blk,
                                                             d_out, d_pair_out);
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}

// <c_2s c_2s+1 c_2t c_2t+1> of every chain and link into d_out [n][n_links]
// and/or its per-pair parts into d_pairs [n][n_links][K][K] (device; either
// may be null).
ggf_status ggf_fermion4(ggf_ctx* ctx, cxd* d_out, cudaStream_t st, cxd* d_pairs) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    GGF_TRY(ggf_flush(ctx, st));
    const int ng = OT / g.B, bpc = (g.n_links + ng - 1) / ng;
    const long long blocks = (long long)bpc * ch.n;
    if (blocks > 0x7fffffffLL) return ggf_fail(ctx, GGF_EINVAL, "too many chains for one launch");
    const bool fp64 = ch.opts.precision == GGF_FP64;
    const cxd* ready = ggf_obs_weights(ctx, blocks, st);
#define GGF_F4(RW, CW, BW)                                                                                  \
    fermion4_kernel<RW, CW, BW><<<(unsigned)blocks, OT, 0, st>>>(ctx->dc(), bpc, (const RW*)ch.Wr,           \
                                                                 (const CW*)ch.Wc, ch.ell, ready, d_out, d_pairs)
    if (g.B == 8) {
        if (fp64) GGF_F4(double, cxd, 8); else GGF_F4(float, cxf, 8);
    } else if (g.B == 16) {
        if (fp64) GGF_F4(double, cxd, 16); else GGF_F4(float, cxf, 16);
    } else {
        return ggf_fail(ctx, GGF_EINVAL, "n_v must be 1 or 2");
    }
#undef GGF_F4
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}

// Site and link bilinears of every chain into d_site [n][V] and d_link
// [n][n_links][2][2], and their per-pair parts into d_pair_site [n][V][K][K]
// and d_pair_link [n][n_links][2][2][K][K] (device; any may be null).
ggf_status ggf_fermion(ggf_ctx* ctx, cxd* d_site, cxd* d_link, cxd* d_pair_site, cxd* d_pair_link,
                       cudaStream_t st) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    GGF_TRY(ggf_flush(ctx, st));
    // only the items that an output wants
    const int it0 = d_site || d_pair_site ? 0 : g.V;
    const int items = (d_link || d_pair_link ? g.V + g.n_links : g.V) - it0;
    if (items <= 0) return GGF_OK;
    const int ng = OT / g.B, bpc = (items + ng - 1) / ng;
    const long long blocks = (long long)bpc * ch.n;
    if (blocks > 0x7fffffffLL) return ggf_fail(ctx, GGF_EINVAL, "too many chains for one launch");
    const bool fp64 = ch.opts.precision == GGF_FP64;
    const cxd* ready = ggf_obs_weights(ctx, blocks, st);
#define GGF_FE(RW, CW, BW)                                                                                       \
    fermion_kernel<RW, CW, BW><<<(unsigned)blocks, OT, 0, st>>>(ctx->dc(), bpc, it0, items, (const RW*)ch.Wr,     \
                                                                (const CW*)ch.Wc, ch.ell, ready, d_site, d_link,         \
                                                                d_pair_site, d_pair_link)
    if (g.B == 8) {
        if (fp64) GGF_FE(double, cxd, 8); else GGF_FE(float, cxf, 8);
    } else if (g.B == 16) {
        if (fp64) GGF_FE(double, cxd, 16); else GGF_FE(float, cxf, 16);
    } else {
        return ggf_fail(ctx, GGF_EINVAL, "n_v must be 1 or 2");
    }
#undef GGF_FE
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}
