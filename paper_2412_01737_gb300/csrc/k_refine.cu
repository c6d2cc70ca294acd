// Newton refinement of an FP32 inverse W ~ M_nm(G)^{-1} (the periodic refresh
// of the cached inverses of FP32 chains):
//     R = I - M W,     W <- W + W R.
// M is sparse (each row couples a virtual Majorana to its own site and to
// the partner end of its link, <= B + 2 n_v entries), so R costs O(N^2 B)
// FP32 work assembled from the links; the dense product W R runs on the
// tcgen05 tensor cores through the flush kernel (W -= U V with U = W and
// V = -R, rank N).  The error of W after a step is about ||R||^2 plus the
// FP32 floor of computing R; for a residual below 1e-4 one TF32 product per
// term suffices (its 2^-11 rounding of a correction that small is below the
// FP32 rounding of W), larger residuals take the three-product split.
//
// Matrices are refined in batches (of one family, from any chains): one
// residual launch, one read-back of the largest residuals and one product
// launch for all of them.  One matrix at a time, a refresh of 1 023 chains of
// 8 x 8 Z2 (N = 512) took 74 ms of kernels of 10 to 49 us that left most of
// the chip idle, and 37 ms of gaps between them; in batches about 6 ms together.
#include <algorithm>
#include <vector>
#include "ggf_ctx.h"
#include "ggf_geom.cuh"

ggf_status ggf_flush_tc_items(ggf_ctx* ctx, bool cplx, int n, float* W, const int* wmap, const float* Pan,
                              const int* pend, int terms, unsigned char* ps, cudaStream_t st);
size_t ggf_flush_ps_item_bytes(ggf_ctx* ctx, bool cplx);

namespace {

constexpr int RB = 8;          // output rows per CTA (one panel chunk)
constexpr int RT = 256;        // columns per CTA
constexpr int MAXC = 64;       // distinct columns of M touched by RB rows

template <class T> struct RefTy;
template <> struct RefTy<double> { typedef float S; };
template <> struct RefTy<cxd> { typedef cxf S; };

__device__ __forceinline__ float to_s(double v) { return (float)v; }
__device__ __forceinline__ cxf to_s(cxd v) { return {(float)v.x, (float)v.y}; }

// V^T panels (chunk-major, row = output column j, rank = output row q) of
// -R = M W - I for rows q0 .. q0 + 7 of every item (grid.y) with act != 0: the
// matrix M of (cfg, pair) and block wmap of W; the largest |R| entry goes to
// rmax[item] (float bits, non-negative values compare as ints).  The
// coefficients of the eight rows (FP64 twists) are formed once and serve every
// column block.
template <class T>
__global__ void __launch_bounds__(RT) resid_kernel(DevConst dc, const void* links, const int* cfgs, const int* pairs,
                                                   const int* wmap, const int* act, const float* Wbase, float* Pan,
                                                   size_t NK, int NP, unsigned* rmax) {
    typedef typename RefTy<T>::S S;
    constexpr bool CPLX = Sc<T>::CPLX;
    __shared__ int cols[MAXC];
    __shared__ S coef[RB][MAXC];
    __shared__ int ncol;
    __shared__ float red[RT / 32];
    const Geometry& g = dc.g;
    const int N = g.N, B = g.B, item = blockIdx.y;
    if (!act[item]) return;
    const int cfg = cfgs[item], pair = pairs[item];
    const float* W = Wbase + (size_t)wmap[item] * N * N * (CPLX ? 2 : 1);
    float* Vt = Pan + ((size_t)item * 2 + 1) * (CPLX ? 2 : 1) * NK;
    const int q0 = blockIdx.x * RB;
    if (threadIdx.x == 0) {
        // columns: the site of q0 .. q0 + 7, then the partner ends of their links
        int n = 0;
        const int s = q0 / B;
        for (int k = 0; k < B; ++k) cols[n++] = s * B + k;
        for (int r = 0; r < RB; ++r) {
            const int q = q0 + r;
            if (q >= N) break;
            // the other end of q's link: the end e ^ 1 of the neighbouring site
            const int e = (q % B) / g.h2, d = e >> 1;
            const int x = s % g.L, y = s / g.L;
            int ps;
            if (e & 1) ps = d == 0 ? y * g.L + (x + 1) % g.L : ((y + 1) % g.L) * g.L + x;
            else ps = d == 0 ? y * g.L + (x + g.L - 1) % g.L : ((y + g.L - 1) % g.L) * g.L + x;
            const int pe = e ^ 1;
            for (int k = 0; k < g.h2; ++k) {
                const int c = ps * B + pe * g.h2 + k;
                bool dup = false;
                for (int z = 0; z < n; ++z) dup |= cols[z] == c;
                if (!dup && n < MAXC) cols[n++] = c;
            }
        }
        ncol = n;
    }
    __syncthreads();
    const int nc = ncol;
    for (int e = threadIdx.x; e < RB * nc; e += RT) {
        const int r = e / nc, c = e - r * nc;
        const int q = q0 + r;
        coef[r][c] = q < N ? to_s(assemble_elem<T>(dc, links, cfg, pair, q, cols[c])) : to_s(Sc<T>::zero());
    }
    __syncthreads();
    float mx = 0.f;
    for (int j = threadIdx.x; j < N; j += RT) {
        S acc[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) acc[r] = S{};
        for (int c = 0; c < nc; ++c) {
            if (!CPLX) {
                const float w = W[(size_t)cols[c] * N + j];
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    float& a = *(float*)&acc[r];
                    a = fmaf(*(const float*)&coef[r][c], w, a);
                }
            } else {
                const float2 w = *(const float2*)(W + ((size_t)cols[c] * N + j) * 2);
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    cxf& a = *(cxf*)&acc[r];
                    const cxf m = *(const cxf*)&coef[r][c];
                    a.x = fmaf(m.x, w.x, a.x);
                    a.x = fmaf(-m.y, w.y, a.x);
                    a.y = fmaf(m.x, w.y, a.y);
                    a.y = fmaf(m.y, w.x, a.y);
                }
            }
        }
        float out_r[RB], out_i[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const int q = q0 + r;
            if (!CPLX) {
                float v = *(float*)&acc[r];
                if (q == j) v -= 1.f;
                out_r[r] = v;
                out_i[r] = 0.f;
                mx = (v == v) ? fmaxf(mx, fabsf(v)) : __int_as_float(0x7f800000);
            } else {
                cxf v = *(cxf*)&acc[r];
                if (q == j) v.x -= 1.f;
                out_r[r] = v.x;
                out_i[r] = v.y;
                mx = (v.x == v.x && v.y == v.y) ? fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y))) : __int_as_float(0x7f800000);
            }
            if (q >= N) { out_r[r] = 0.f; out_i[r] = 0.f; }
        }
        float* dst = Vt + pidx(j, q0, NP);
        *(float4*)dst = make_float4(out_r[0], out_r[1], out_r[2], out_r[3]);
        *(float4*)(dst + 4) = make_float4(out_r[4], out_r[5], out_r[6], out_r[7]);
        if (CPLX) {
            float* di = dst + NK;
            *(float4*)di = make_float4(out_i[0], out_i[1], out_i[2], out_i[3]);
            *(float4*)(di + 4) = make_float4(out_i[4], out_i[5], out_i[6], out_i[7]);
        }
    }
    if (!(mx == mx)) mx = __int_as_float(0x7f800000);   // NaN -> +inf
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int w = 0; w < RT / 32; ++w) m = fmaxf(m, red[w]);
        atomicMax(rmax + item, __float_as_uint(m));
    }
}

// U panels = W of the items with pend != 0: element (row i, rank q) <- W[i][q], eight rank columns per thread
template <bool CPLX>
__global__ void upanel_kernel(int N, const int* wmap, const int* pend, const float* Wbase, float* Pan, size_t NK, int NP) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int q0 = blockIdx.y * 8, item = blockIdx.z;
    if (i >= N || !pend[item]) return;
    const float* W = Wbase + (size_t)wmap[item] * N * N * (CPLX ? 2 : 1);
    float* U = Pan + (size_t)item * 2 * (CPLX ? 2 : 1) * NK;
    float* dst = U + pidx(i, q0, NP);
    if (!CPLX) {
        const float* src = W + (size_t)i * N + q0;
        *(float4*)dst = *(const float4*)src;
        *(float4*)(dst + 4) = *(const float4*)(src + 4);
    } else {
        const float4* src = (const float4*)(W + ((size_t)i * N + q0) * 2);
        float re[8], im[8];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float4 v = src[t];
            re[2 * t] = v.x; im[2 * t] = v.y; re[2 * t + 1] = v.z; im[2 * t + 1] = v.w;
        }
        *(float4*)dst = make_float4(re[0], re[1], re[2], re[3]);
        *(float4*)(dst + 4) = make_float4(re[4], re[5], re[6], re[7]);
        *(float4*)(dst + NK) = make_float4(im[0], im[1], im[2], im[3]);
        *(float4*)(dst + NK + 4) = make_float4(im[4], im[5], im[6], im[7]);
    }
}

}  // namespace

// ---- batches of matrices of one family -----------------------------------------

namespace {

size_t panel_bytes(int N, bool cplx) { return panel_plane(N, N) * (cplx ? 4 : 2) * sizeof(float); }

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

// Plans a batch of at most `items` matrices: their number (at least one), the
// workspace they need, and whether their pre-split operands go into the
// chains' flush scratch (idle outside a sweep) or into the workspace.  A batch
// makes the workspace no larger than 1 GiB and a quarter of the free memory
// (one matrix is always taken); a workspace that is larger already is used whole.
void ggf_refine_plan(ggf_ctx* ctx, bool cplx, int items, RefineBatch& b) {
    const int N = ctx->g.N;
    const Chains& ch = ctx->ch;
    const size_t pb = panel_bytes(N, cplx), psb = ggf_flush_ps_item_bytes(ctx, cplx);
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    const size_t budget = std::max(ctx->work_bytes, std::min<size_t>((size_t)1 << 30, free_b / 4));
    b.cplx = cplx;
    size_t n;
    if (ch.ps && psb <= ch.ps_bytes) {
        n = std::min(ch.ps_bytes / psb, budget / pb);
        b.own_ps = false;
        b.ps = ch.ps;
    } else {
        n = budget / (pb + psb);
        b.own_ps = n > 0;
        b.ps = nullptr;                        // n = 0: operands are split per tile
    }
    b.cap = (int)std::max<size_t>(1, std::min<size_t>({n, (size_t)items, (size_t)32768}));
    b.bytes = up256(pb * b.cap) + (b.own_ps ? up256(psb * b.cap) : 0) + 5 * up256((size_t)b.cap * sizeof(int));
}

// Lays the batch out in ws (b.bytes) and uploads its items: configuration and
// pair of M, block of W.
ggf_status ggf_refine_begin(ggf_ctx* ctx, RefineBatch& b, int n, const int* cfg, const int* pair, const int* block,
                            float* W, void* ws, cudaStream_t st) {
    const int N = ctx->g.N;
    unsigned char* q = (unsigned char*)ws;
    auto take = [&](size_t bytes) { unsigned char* p = q; q += up256(bytes); return p; };
    b.n = n;
    b.W = W;
    b.Pan = (float*)take(panel_bytes(N, b.cplx) * b.cap);
    if (b.own_ps) b.ps = take(ggf_flush_ps_item_bytes(ctx, b.cplx) * b.cap);
    const size_t ib = (size_t)b.cap * sizeof(int);
    b.d_cfg = (int*)take(ib);
    b.d_pair = (int*)take(ib);
    b.d_block = (int*)take(ib);
    b.d_pend = (int*)take(ib);
    b.d_rmax = (unsigned*)take(ib);
    GGF_CK(cudaMemcpyAsync(b.d_cfg, cfg, n * sizeof(int), cudaMemcpyHostToDevice, st));
    GGF_CK(cudaMemcpyAsync(b.d_pair, pair, n * sizeof(int), cudaMemcpyHostToDevice, st));
    GGF_CK(cudaMemcpyAsync(b.d_block, block, n * sizeof(int), cudaMemcpyHostToDevice, st));
    return GGF_OK;
}

// max |I - M W| of the items with act[i] != 0 into rmax[i]; keeps their -R =
// M W - I for the next product.  Synchronises the stream.
ggf_status ggf_refine_measure(ggf_ctx* ctx, RefineBatch& b, const void* d_links, const std::vector<int>& act,
                              std::vector<double>& rmax, cudaStream_t st) {
    const int N = ctx->g.N, NP = panel_rows(N);
    const size_t NK = panel_plane(N, N);
    GGF_CK(cudaMemcpyAsync(b.d_pend, act.data(), b.n * sizeof(int), cudaMemcpyHostToDevice, st));
    GGF_CK(cudaMemsetAsync(b.d_rmax, 0, b.n * sizeof(unsigned), st));
    dim3 grid((N + RB - 1) / RB, b.n);
    if (b.cplx)
        resid_kernel<cxd><<<grid, RT, 0, st>>>(ctx->dc(), d_links, b.d_cfg, b.d_pair, b.d_block, b.d_pend, b.W, b.Pan, NK,
                                               NP, b.d_rmax);
    else
        resid_kernel<double><<<grid, RT, 0, st>>>(ctx->dc(), d_links, b.d_cfg, b.d_pair, b.d_block, b.d_pend, b.W, b.Pan,
                                                  NK, NP, b.d_rmax);
    GGF_CK(cudaGetLastError());
    ctx->launches += 1;
    std::vector<float> h(b.n);
    GGF_CK(cudaMemcpyAsync(h.data(), b.d_rmax, b.n * sizeof(float), cudaMemcpyDeviceToHost, st));
    GGF_CK(cudaStreamSynchronize(st));
    for (int i = 0; i < b.n; ++i)
        if (act[i]) rmax[i] = h[i];
    return GGF_OK;
}

// W <- W + W R of the items with act[i] != 0, with the R of the last measure:
// one TF32 product, or (terms = 3) the FP32-accurate three-product split.
ggf_status ggf_refine_apply(ggf_ctx* ctx, RefineBatch& b, const std::vector<int>& act, int terms, cudaStream_t st) {
    const int N = ctx->g.N, NP = panel_rows(N);
    if (N % 8) return ggf_fail(ctx, GGF_EINVAL, "refinement needs N divisible by 8");
    const size_t NK = panel_plane(N, N);
    std::vector<int> pend(b.n);
    for (int i = 0; i < b.n; ++i) pend[i] = act[i] ? N / 8 : 0;
    GGF_CK(cudaMemcpyAsync(b.d_pend, pend.data(), b.n * sizeof(int), cudaMemcpyHostToDevice, st));
    dim3 ug((N + 255) / 256, N / 8, b.n);
    if (b.cplx) upanel_kernel<true><<<ug, 256, 0, st>>>(N, b.d_block, b.d_pend, b.W, b.Pan, NK, NP);
    else upanel_kernel<false><<<ug, 256, 0, st>>>(N, b.d_block, b.d_pend, b.W, b.Pan, NK, NP);
    GGF_CK(cudaGetLastError());
    ctx->launches += 3;
    GGF_TRY(ggf_flush_tc_items(ctx, b.cplx, b.n, b.W, b.d_block, b.Pan, b.d_pend, terms, b.ps, st));
    GGF_CK(cudaStreamSynchronize(st));     // pend is read by the copy above
    return GGF_OK;
}
