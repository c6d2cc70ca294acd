// Score of the site blocks: d log N(G) / d D_s for every chain and site, from
// the chains' inverses (score_entry in ggf_obs_group.cuh).
// With it the gradient of a Wilson-loop energy with respect to the site
// parameters is the covariance E_p[(W(G) - E) sum_s tr(S_s^T dD_s)].
//
// What bounds them: the outputs' writes and the latency of the block loads; 32
// chains of 8 x 8 U(1), K = 2: site scores 398 us with one thread per site that
// summed into global memory, 27 with one thread per entry; link scores 147
// us with one thread per (pair, link), 60 with a warp; 1024 chains of 8 x 8
// Z2 94 -> 44 and 294 -> 135 us (320 and 288 with the weights formed in every CTA).
#include "ggf_obs_group.cuh"

namespace {

// One CTA per (chain, site), one thread per entry: thread (j, i) reads
// W_p[s B + j][s B + i], so that a row of the block is one run, and the sums
// are transposed through shared memory into out[i][j].
template <class RW, class CW, int B>
__global__ void __launch_bounds__(B * B) score_kernel(DevConst dc, const RW* Wr, const CW* Wc, const cxd* ell,
                                                      const cxd* ready, double* out) {
    __shared__ double tr[B][B + 1];
    __shared__ PairWeights pw;
    const int c = blockIdx.x / dc.g.V, s = blockIdx.x % dc.g.V, j = threadIdx.x / B, i = threadIdx.x % B;
    chain_weights(dc, c, ell, ready, pw);
    const double acc = score_entry<RW, CW, B>(dc, c, s, i, j, Wr, Wc, pw.E);
    tr[i][j] = acc;
    __syncthreads();
    out[(size_t)blockIdx.x * B * B + threadIdx.x] = tr[threadIdx.x / B][threadIdx.x % B];
}

// One warp per (chain, pair, link); CTAs stay within a chain.
template <class T, int R>
__device__ __forceinline__ void link_score_warp(const DevConst& dc, const T* W, int l, cxd f, const double* O, cxd* w,
                                                cxd* o) {
    const int lane = threadIdx.x & 31;
    LinkScoreRow<R> m;
    link_score_load<T, R>(dc, W, l, lane, w);
    __syncwarp();
    link_score_mix<R>(O, w, lane, m);
    __syncwarp();
    link_score_put<R>(lane, m, w);
    __syncwarp();
    link_score_out<R>(O, w, f, lane, o);
}

template <class RW, class CW, int R>
__global__ void __launch_bounds__(OT) link_score_kernel(DevConst dc, int blocks_per_chain, const void* links,
                                                        const RW* Wr, const CW* Wc, const cxd* ell, const cxd* ready,
                                                        cxd* out) {
    constexpr int NW = OT / 32, H = R / 2;
    __shared__ PairWeights pw;
    __shared__ cxd blk[NW][R * R];
    __shared__ double Os[NW][H * H];
    const Geometry& g = dc.g;
    const int c = blockIdx.x / blocks_per_chain, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int item = (blockIdx.x - c * blocks_per_chain) * NW + warp;
    chain_weights(dc, c, ell, ready, pw);
    if (item >= dc.P * g.n_links) return;
    const int p = item / g.n_links, l = item % g.n_links;
    link_score_twist<H>(dc, links, c, l, lane, Os[warp]);
    __syncwarp();
    const size_t NN = (size_t)g.N * g.N;
    const cxd f = 0.5 * pw.E[p];
    cxd* o = out + (((size_t)c * dc.P + p) * g.n_links + l) * R * R;
    if (p < dc.K) link_score_warp<RW, R>(dc, Wr + ((size_t)c * dc.K + p) * NN, l, f, Os[warp], blk[warp], o);
    else link_score_warp<CW, R>(dc, Wc + ((size_t)c * dc.Kc + (p - dc.K)) * NN, l, f, Os[warp], blk[warp], o);
}

}  // namespace

ggf_status ggf_flush(ggf_ctx* ctx, cudaStream_t st);

// Link-block scores of every chain, pair and link into d_out
// [n_chains][P][n_links][r][r] (device, complex).
ggf_status ggf_link_score(ggf_ctx* ctx, cxd* d_out, cudaStream_t st) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    GGF_TRY(ggf_flush(ctx, st));
    const int nw = OT / 32, bpc = (ctx->P * g.n_links + nw - 1) / nw;
    const long long blocks = (long long)bpc * ch.n;
    if (blocks > 0x7fffffffLL) return ggf_fail(ctx, GGF_EINVAL, "too many chains for one launch");
    const bool fp64 = ch.opts.precision == GGF_FP64;
    const cxd* ready = ggf_obs_weights(ctx, blocks, st);
#define GGF_LS(RW, CW, R_)                                                                                    \
    link_score_kernel<RW, CW, R_><<<(unsigned)blocks, OT, 0, st>>>(ctx->dc(), bpc, ch.links, (const RW*)ch.Wr, \
                                                                   (const CW*)ch.Wc, ch.ell, ready, d_out)
    if (g.r == 4) {
        if (fp64) GGF_LS(double, cxd, 4); else GGF_LS(float, cxf, 4);
    } else if (g.r == 8) {
        if (fp64) GGF_LS(double, cxd, 8); else GGF_LS(float, cxf, 8);
    } else {
        return ggf_fail(ctx, GGF_EINVAL, "n_v must be 1 or 2");
    }
#undef GGF_LS
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}

// Site scores of every chain into d_out [n_chains][V][B][B] (device, FP64).
ggf_status ggf_score(ggf_ctx* ctx, double* d_out, cudaStream_t st) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    GGF_TRY(ggf_flush(ctx, st));
    const long long blocks = (long long)ch.n * g.V;
    if (blocks > 0x7fffffffLL) return ggf_fail(ctx, GGF_EINVAL, "too many chains for one launch");
    const bool fp64 = ch.opts.precision == GGF_FP64;
    const cxd* ready = ggf_obs_weights(ctx, blocks, st);
#define GGF_SC(RW, CW, B_)                                                                                     \
    score_kernel<RW, CW, B_><<<(unsigned)blocks, B_ * B_, 0, st>>>(ctx->dc(), (const RW*)ch.Wr, (const CW*)ch.Wc, \
                                                                   ch.ell, ready, d_out)
    if (g.B == 8) {
        if (fp64) GGF_SC(double, cxd, 8); else GGF_SC(float, cxf, 8);
    } else if (g.B == 16) {
        if (fp64) GGF_SC(double, cxd, 16); else GGF_SC(float, cxf, 16);
    } else {
        return ggf_fail(ctx, GGF_EINVAL, "n_v must be 1 or 2");
    }
#undef GGF_SC
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}
