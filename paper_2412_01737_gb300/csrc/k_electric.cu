// Electric-field observables (Sec. 5.3), evaluated for every chain and link
// from the inverses W_nm = M_nm(G)^{-1} the sampler keeps:
//   f_E(G)_l = sum_nm lambda_n^* lambda_m <psi_n(G)| I_l |psi_m(G)>_ket / N(G),
// with the insertion I_l acting on the ket's source-end modes of link l (the
// end that carries the twist) before the contraction:
//   Z2:   I_l = the parity of those modes, so that the ket becomes psi_m(G^(l))
//         (the flip X_l of the link, of which the Z2 electric term is a
//         linear function);
//   U(1): I_l = Q_l^2, Q_l = sum_j q_j n_j the twist charge of those modes: the
//         ket depends on its link angle through exp(i theta Q_l), so the
//         single-link integral with <G|J^2|g; G> (J = -i d/dtheta) is
//         -d^2/dtheta^2 of the overlap, i.e. the insertion of Q_l^2;
//   SU(2): I_l = sum_a (Q^a)^2 on the source doublet, Q^a = psi^dag (sigma_a / 2)
//         psi (right translations of the link act on the twist as
//         exp(i eps Q^a)), which is (3/4)(n_0 + n_1 - 2 n_0 n_1).
// The U(1) field <J_l> itself inserts I_l = Q_l (one derivative of the
// overlap), R_nm = sum_j q_j <n_j>; with charge-conserving site tensors and
// neutral bond pairs it obeys Gauss's law configuration by configuration.
// Wick's theorem on the Gaussian operator composed of the sites' virtual
// state and the bond operator X_nm gives the insertion's normalised
// expectation from the covariance of that operator on the end's 2 n_v
// Majoranas S,
//   Gamma_O = i 1 - (1 + i D) W_nm (1 + i Gamma_tw),   G = Gamma_O[S, S],
//   Z2:   R_nm = (-1)^{n_v} Pf(G),
//   SU(2): R_nm = (3/4)(<n_0> + <n_1> - 2 <n_0 n_1>),
//   U(1): R_nm = sum_j q_j^2 <n_j> + 2 sum_{j<k} q_j q_k <n_j n_k>,
//         <n_j> = (1 + G_{2j,2j+1}) / 2,
//         <n_j n_k> = (1 + G_{2j,2j+1} + G_{2k,2k+1} + Pf G[2j, 2j+1, 2k, 2k+1]) / 4,
// with M_nm = D + Gamma_tw, D the sites' virtual blocks and Gamma_tw =
// O(G) Gamma_X O(G)^T the twisted link blocks.  D is block diagonal by site
// and Gamma_tw by link, so [(1 + i D) W (1 + i Gamma_tw)]_SS involves only the
// B x r block of W between the source site's virtual Majoranas and the link's
// r Majoranas.  D and the twist are real and Gamma_X of (m, n) is the complex
// conjugate of that of (n, m), so M_mn = conj(M_nm): both orders of a pair
// n < m come from its one stored inverse.  With N_nm = e^{logc + ell}
// (N_mn = conj N_nm) and the pair weights of the sampler's combination,
//   f_E(G)_l = sum_nm lambda_n^* lambda_m N_nm R_nm / sum_nm lambda_n^* lambda_m N_nm.
//
// What bounds it: latency of short dependent phases (load a block, two small
// products, the insertion) over many independent items; 32 chains of 8 x 8
// U(1), K = 2 took 508 us with one thread per (chain, link) and take 85
// with a group of B lanes (ggf_obs_group.cuh).  Where the chains fill the chip,
// the FP64 unit, 83 % busy: 1024 chains of 8 x 8 Z2 take 99 us, of U(1) 129 (95
// and 122 with one thread per item; 148 for Z2 with the weights formed in every
// CTA and complex products for the real pairs).
#include "ggf_obs_group.cuh"

namespace {

// CTAs of an observable kernel above which the pair weights are formed once per
// chain ahead of it: a launch of about 2 us against some hundred FP64
// instructions per CTA.  Microseconds, in the CTAs and ahead of them: 1024 CTAs
// 21 and 23 (128 chains of 8 x 8 Z2, electric), 19 and 19 (16 of 8 x 8 U(1),
// K = 2, site scores); 2048 CTAs 38 and 34 (256 of 8 x 8 Z2, electric), 32 and 27
// (32 of 8 x 8 U(1), K = 2, site scores); 65536 CTAs 305 and 46 (1024 of 8 x 8 Z2,
// site scores).
constexpr long long OBS_WEIGHTS_ABOVE = 1024;

// A group of B = 4 H lanes per (chain, link); FIELD: the U(1) electric field
// instead of J^2.
template <class RW, class CW, int H, bool FIELD>
__global__ void __launch_bounds__(OT) electric_kernel(DevConst dc, int blocks_per_chain, const void* links, const RW* Wr,
                                                      const CW* Wc, const cxd* ell, const cxd* ready, cxd* out,
                                                      cxd* pair_out) {
    constexpr int B = 4 * H, NG = OT / B;
    __shared__ ElectricShared<H> shared[NG];
    __shared__ PairWeights pw;
    const Geometry& g = dc.g;
    const int c = blockIdx.x / blocks_per_chain, grp = threadIdx.x / B, lane = threadIdx.x % B;
    const int want = (blockIdx.x - c * blocks_per_chain) * NG + grp;
    const int l = min(want, g.n_links - 1);            // idle groups repeat the last link and write nothing
    const bool live = want < g.n_links;
    ElectricShared<H>& sh = shared[grp];
    const double gval = electric_link(g, links, c, l);
    // the twists of all the CTA's links by the second warp, beside the weights
    const int modes = electric_modes(g);
    if (threadIdx.x >= 32 && threadIdx.x < 32 + NG * modes) {
        const int i = threadIdx.x - 32, of = i / modes;
        electric_twist<H>(g, links, c, min(want - grp + of, g.n_links - 1), i - of * modes, shared[of]);
    }
    chain_weights(dc, c, ell, ready, pw);
    const int K = dc.K;
    const size_t NN = (size_t)g.N * g.N;
    cxd num = {0.0, 0.0};
    cxd* po = pair_out ? pair_out + ((size_t)c * g.n_links + l) * K * K : nullptr;
    for (int p = 0; p < dc.P; ++p) {
        const bool cplx = p >= K;
        const cxd v = cplx ? electric_pair<CW, H, FIELD>(dc, p - K, l, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, lane, gval, sh)
                           : electric_pair<RW, H, FIELD>(dc, p, l, Wr + ((size_t)c * K + p) * NN, lane, gval, sh);
        electric_term(dc, p, lane, live, pw.np[p], pw.E[p], v, num, po);
    }
    if (dc.Kc > 0) num = num + shfl_xor_(num, 1);
    if (out && live && lane == 0) out[(size_t)c * g.n_links + l] = num;
}

// A group of G lanes per chain, the smallest power of two that holds the pairs
// (an FP64 instruction costs a warp the same whatever the number of its lanes):
// out [n][2][P].
__global__ void __launch_bounds__(OT) obs_weights_kernel(DevConst dc, int n_chains, int G, const cxd* ell, cxd* out) {
    const int want = (blockIdx.x * OT + threadIdx.x) / G, c = min(want, n_chains - 1);
    cxd* o = out + (size_t)c * 2 * dc.P;
    warp_weights(dc, ell + (size_t)c * dc.P, G, want < n_chains, o, o + dc.P);
}

// One thread per chain.
__global__ void pair_norm_kernel(DevConst dc, int n_chains, const cxd* ell, cxd* out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_chains) return;
    pair_norm_item(dc, c, ell, out);
}

}  // namespace

ggf_status ggf_flush(ggf_ctx* ctx, cudaStream_t st);

// The chains' pair weights for an observable kernel of `blocks` CTAs, formed
// once per chain ahead of it, or null where its CTAs form their chain's
// themselves (OBS_WEIGHTS_ABOVE).
const cxd* ggf_obs_weights(ggf_ctx* ctx, long long blocks, cudaStream_t st) {
    const Chains& ch = ctx->ch;
    if (blocks <= OBS_WEIGHTS_ABOVE) return nullptr;
    int G = 1;
    while (G < 32 && G < ctx->P) G *= 2;
    obs_weights_kernel<<<(unsigned)(((long long)ch.n * G + OT - 1) / OT), OT, 0, st>>>(ctx->dc(), ch.n, G, ch.ell,
                                                                                        ch.obs_w);
    return ch.obs_w;
}

// N_nm(G) / N(G) of every chain into d_out [n_chains][K][K] (device).
ggf_status ggf_pair_norm(ggf_ctx* ctx, cxd* d_out, cudaStream_t st) {
    Chains& ch = ctx->ch;
    pair_norm_kernel<<<(ch.n + 127) / 128, 128, 0, st>>>(ctx->dc(), ch.n, ch.ell, d_out);
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}

// f_E for every chain and link into d_out [n_chains][n_links] and/or its
// per-pair parts into d_pairs [n_chains][n_links][K][K] (device; either may
// be null): Z2 the flip, U(1) and SU(2) the Casimir J^2.
ggf_status ggf_electric(ggf_ctx* ctx, cxd* d_out, cxd* d_pairs, cudaStream_t st, bool field) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    // pending delayed updates first, so that W is the inverse at the current links
    GGF_TRY(ggf_flush(ctx, st));
    const int ng = OT / g.B, bpc = (g.n_links + ng - 1) / ng;
    const long long blocks = (long long)bpc * ch.n;
    if (blocks > 0x7fffffffLL) return ggf_fail(ctx, GGF_EINVAL, "too many chains for one launch");
    const bool fp64 = ch.opts.precision == GGF_FP64;
    const void* lk = ch.links;
    const cxd* ready = ggf_obs_weights(ctx, blocks, st);
#define GGF_EL2(RW, CW, H, F)                                                                                       \
    electric_kernel<RW, CW, H, F><<<(unsigned)blocks, OT, 0, st>>>(ctx->dc(), bpc, lk, (const RW*)ch.Wr,             \
                                                                   (const CW*)ch.Wc, ch.ell, ready, d_out, d_pairs)
#define GGF_EL(RW, CW, H)                  \
    do {                                   \
        if (field) GGF_EL2(RW, CW, H, true); \
        else GGF_EL2(RW, CW, H, false);      \
    } while (0)
    if (g.h2 == 2) {
        if (fp64) GGF_EL(double, cxd, 2); else GGF_EL(float, cxf, 2);
    } else if (g.h2 == 4) {
        if (fp64) GGF_EL(double, cxd, 4); else GGF_EL(float, cxf, 4);
    } else {
        return ggf_fail(ctx, GGF_EINVAL, "n_v must be 1 or 2");
    }
#undef GGF_EL
#undef GGF_EL2
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}
