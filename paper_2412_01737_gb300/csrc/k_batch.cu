// Batched (submatrix) delayed updates for local Metropolis sweeps
// (Sec. 5.1 sampling of p(G); the blocking of the Sherman-Morrison-Woodbury
// updates is this library's design, not the paper's).
//
// A batch is kb consecutive links l0 .. l0 + kb - 1 of the sweep order.  Every
// link end belongs to exactly one link, so the batch's Majorana sets S_j are
// disjoint and T = S_0 u ... u S_{kb-1} has exactly kb r elements (position
// j r + xi of T is Majorana xi of link l0 + j).  Every proposal of the batch
// needs only the block of the current inverse on T.  With W the inverse at
// the start of the batch, C = W[:, T], Y = W[T, :], G0 = W[T, T]:
//   batch_gather  C -> U panel, Y^T -> V^T panel, G := G0 (C read as
//                 the true columns: -Y^T, equal in exact arithmetic, makes
//                 the rounding error grow geometrically)
//   batch_steps   one cluster per chain (k_steps.cu) runs the kb link steps on
//                 the small matrices, from X = 0: ratio from G[S_j, S_j], decision, and on accept,
//                 with Z = (1 + Delta G[S, S])^{-1} Delta,
//                   G[F, F] -= G[F, S] Z G[S, F]   (F: the later links' rows)
//                   X       += P Z Q,  P = E_S - X G0[:, S],
//                                      Q = E_S^T - G0[S, :] X,
//                 so that the exact inverse after the batch is W - C X Y
//                 (each step is the rank-r update W' = W - W[:, S] Z W[S, :]
//                 with W[:, S] = C P and W[S, :] = Q Y).
//   batch_apply   V^T <- V^T X^T  (V = X Y)
// followed by the flush W <- W - U V (tcgen05 tensor cores for FP32 chains).
// Per batch and pair this reads C and Y once (2 N kb r elements) instead of
// two N-long panel products per accepted link, and folds kb links into one
// pass over W.
#include "ggf_sweep.cuh"

// 1: the X product of FP32 batches runs on the tensor cores (k_apply_tc.cu)
#ifndef GGF_APPLY_TC
#define GGF_APPLY_TC 1
#endif

namespace {

// ---- gather -------------------------------------------------------------------
// Grid (ceil(N / BR), family pairs, chains), 256 threads.  Rows i0 .. i0+BR-1
// of the U panel (C = W[:, T]) and of the V^T panel (Y^T = W[T, :]^T); the
// rows of G := W[T, T] whose T index falls in the block.
template <class T>
__global__ void __launch_bounds__(256) batch_gather(Geometry g, int l0, int kb, int fam_pairs, int KRM, int BR,
                                                    const T* W, typename Sc<T>::R* Pan, T* Sm) {
    typedef typename Sc<T>::R RR;
    const int c = blockIdx.z, p = blockIdx.y, N = g.N, r = g.r, kr = kb * r;
    extern __shared__ unsigned char smraw[];
    int* Tl = (int*)smraw;                                   // [kr]
    T* tile = (T*)(smraw + ((kr * sizeof(int) + 15) & ~(size_t)15));   // [BR][kr + 1]
    for (int q = threadIdx.x; q < kr; q += blockDim.x) {
        int a0, b0;
        link_ends(g, l0 + q / r, a0, b0);
        Tl[q] = link_majorana(g, a0, b0, q % r);
    }
    __syncthreads();
    const int i0 = blockIdx.x * BR, nb = min(BR, N - i0), ld = kr + 1;
    const size_t NK = panel_plane(N, KRM), base = (size_t)c * fam_pairs + p;
    const int NP = panel_rows(N);
    const T* Wp = W + base * N * N;
    RR* U = Pan + base * 2 * PanelIO<T>::PLANES * NK;
    RR* Vt = U + PanelIO<T>::PLANES * NK;
    T* Gm = Sm + base * 2 * KRM * KRM;
    // V^T rows: tile[ii][q] = W[T_q][i0 + ii], read along rows of W
    for (int e = threadIdx.x; e < kr * BR; e += blockDim.x) {
        int q = e / BR, ii = e - q * BR;
        tile[ii * ld + q] = ii < nb ? Wp[(size_t)Tl[q] * N + i0 + ii] : Sc<T>::zero();
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nb * kr; e += blockDim.x) {
        int ii = e / kr, q = e - ii * kr;
        PanelIO<T>::st(Vt, NK, pidx(i0 + ii, q, NP), tile[ii * ld + q]);
    }
    __syncthreads();
    // U rows: the true columns W[i0 + ii][T_q].  Replacing them by -Y^T (equal
    // for an exactly antisymmetric W) lets the rounding error grow
    // geometrically from batch to batch.
    for (int e = threadIdx.x; e < nb * kr; e += blockDim.x) {
        int ii = e / kr, q = e - ii * kr;
        T v = Wp[(size_t)(i0 + ii) * N + Tl[q]];
        tile[ii * ld + q] = v;
        PanelIO<T>::st(U, NK, pidx(i0 + ii, q, NP), v);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int a = warp; a < kr; a += nw) {
        const int ii = Tl[a] - i0;
        if (ii < 0 || ii >= nb) continue;
        for (int q = lane; q < kr; q += 32) {
            Gm[(size_t)a * KRM + q] = tile[ii * ld + q];   // W[T_a][T_q] = U[T_a][q]
        }
    }
}

// ---- V^T <- V^T X^T -----------------------------------------------------------
// Grid (ceil(N / RB), family pairs, chains) with RB = 16 RPT rows per CTA,
// 256 threads as 16 x 16.  A CTA stages its RB rows of V^T in shared memory
// and rewrites them in place; per 128-wide output chunk, thread (ty, tx)
// accumulates rows ty RPT .. + RPT - 1 x outputs tx + 16 t (t = 0 .. 7) over
// the rank, with X^T staged 16 columns at a time.  Interleaved outputs make
// the 16 threads of a row read 16 consecutive elements of a staged X^T row
// (contiguous blocks of 8 per thread put them 8 elements apart: 4- to 16-way
// bank conflicts) and write 8 consecutive rank columns of a panel chunk.
constexpr int AP_LDX = 132;   // X^T stage row length (128 outputs + pad, 16-byte rows)

template <class T, int RPT>
__global__ void __launch_bounds__(256) batch_apply(int N, int fam_pairs, int KRM, int kr, typename Sc<T>::R* Pan,
                                                   const T* Sm, const int* pend) {
    typedef typename Sc<T>::R RR;
    constexpr int RB = 16 * RPT;
    const int c = blockIdx.z;
    if (pend[c] == 0) return;
    const int p = blockIdx.y;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int ld = kr + 1;
    T* Xs = (T*)smraw;           // [16][AP_LDX]  X^T chunk: Xs[bb][aa] = X[a0 + aa][b0 + bb]
    T* Vs = Xs + 16 * AP_LDX;    // [RB][kr + 1]
    const size_t NK = panel_plane(N, KRM), base = (size_t)c * fam_pairs + p;
    const int NP = panel_rows(N);
    RR* Vt = Pan + base * 2 * PanelIO<T>::PLANES * NK + PanelIO<T>::PLANES * NK;
    const T* Xm = Sm + base * 2 * KRM * KRM + (size_t)KRM * KRM;
    const int i0 = blockIdx.x * RB, nb = min(RB, N - i0);
    for (int e = threadIdx.x; e < RB * kr; e += blockDim.x) {
        int ii = e / kr, q = e - ii * kr;
        Vs[ii * ld + q] = ii < nb ? PanelIO<T>::ld(Vt, NK, pidx(i0 + ii, q, NP)) : Sc<T>::zero();
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    for (int a0 = 0; a0 < kr; a0 += 128) {
        T acc[RPT][8];
#pragma unroll
        for (int u = 0; u < RPT; ++u)
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[u][t] = Sc<T>::zero();
        // X chunks are loaded into registers one chunk ahead (8 values per
        // thread), so their global loads overlap the previous chunk's products
        T xn[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const int e = threadIdx.x + w * 256, aa = e >> 4, bb = e & 15;
            xn[w] = (a0 + aa < kr && bb < kr) ? Xm[(size_t)(a0 + aa) * KRM + bb] : Sc<T>::zero();
        }
        for (int b0 = 0; b0 < kr; b0 += 16) {
            __syncthreads();
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const int e = threadIdx.x + w * 256;
                Xs[(e & 15) * AP_LDX + (e >> 4)] = xn[w];
            }
            __syncthreads();
            if (b0 + 16 < kr) {
#pragma unroll
                for (int w = 0; w < 8; ++w) {
                    const int e = threadIdx.x + w * 256, aa = e >> 4, bb = b0 + 16 + (e & 15);
                    xn[w] = (a0 + aa < kr && bb < kr) ? Xm[(size_t)(a0 + aa) * KRM + bb] : Sc<T>::zero();
                }
            }
            const int bn = min(16, kr - b0);
            for (int bb = 0; bb < bn; ++bb) {
                T v[RPT], x[8];
#pragma unroll
                for (int u = 0; u < RPT; ++u) v[u] = Vs[(ty * RPT + u) * ld + b0 + bb];
#pragma unroll
                for (int t = 0; t < 8; ++t) x[t] = Xs[bb * AP_LDX + tx + 16 * t];
#pragma unroll
                for (int u = 0; u < RPT; ++u)
#pragma unroll
                    for (int t = 0; t < 8; ++t) acc_add(acc[u][t], v[u], x[t]);
            }
        }
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            const int ii = ty * RPT + u;
            if (ii >= nb) continue;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int aa = a0 + tx + 16 * t;
                if (aa < kr) PanelIO<T>::st(Vt, NK, pidx(i0 + ii, aa, NP), acc[u][t]);
            }
        }
    }
}

size_t apply_smem(int RPT, int kr, size_t tb) { return (16 * AP_LDX + (size_t)16 * RPT * (kr + 1)) * tb; }

int gather_rows(int kr, size_t tb) {
    int br = 32;
    while (br > 4 && (size_t)br * (kr + 1) * tb > 96 * 1024) br >>= 1;
    return br;
}

}  // namespace

ggf_status ggf_flush(ggf_ctx* ctx, cudaStream_t st);
ggf_status ggf_prepare_steps(ggf_ctx* ctx);
bool ggf_steps_fit(ggf_ctx* ctx, int kmax, bool fp64);
ggf_status ggf_batch_steps(ggf_ctx* ctx, int l0, int kb, void* Sr, void* Sc_, cudaStream_t st);
ggf_status ggf_apply_tc(ggf_ctx* ctx, bool cplx, int fam_pairs, int kr, float* Pan, const float* Sm, cudaStream_t st);

// Shared-memory caps of the batch kernels (once per device, like the other
// sampler kernels), and the largest batch that fits.
ggf_status ggf_prepare_batch(ggf_ctx* ctx) {
    static bool done[64] = {false};
    if (ctx->device >= 0 && ctx->device < 64 && done[ctx->device]) return GGF_OK;
    int mx = 0;
    GGF_CK(cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    auto cap = [&](const void* fn) -> ggf_status {
        cudaFuncAttributes fa;
        GGF_CK(cudaFuncGetAttributes(&fa, fn));
        GGF_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, mx - (int)fa.sharedSizeBytes));
        return GGF_OK;
    };
    GGF_TRY(cap((const void*)batch_gather<double>));
    GGF_TRY(cap((const void*)batch_gather<float>));
    GGF_TRY(cap((const void*)batch_gather<cxd>));
    GGF_TRY(cap((const void*)batch_gather<cxf>));
    GGF_TRY(ggf_prepare_steps(ctx));
    GGF_TRY(cap((const void*)batch_apply<double, 4>));
    GGF_TRY(cap((const void*)batch_apply<float, 4>));
    GGF_TRY(cap((const void*)batch_apply<cxd, 4>));
    GGF_TRY(cap((const void*)batch_apply<cxf, 4>));
    GGF_TRY(cap((const void*)batch_apply<double, 2>));
    GGF_TRY(cap((const void*)batch_apply<float, 2>));
    GGF_TRY(cap((const void*)batch_apply<cxd, 2>));
    GGF_TRY(cap((const void*)batch_apply<cxf, 2>));
    if (ctx->device >= 0 && ctx->device < 64) done[ctx->device] = true;
    return GGF_OK;
}

// Shared memory the batch kernels need for batches of kmax links; EINVAL if
// it exceeds the device's per-block limit.
ggf_status ggf_check_batch(ggf_ctx* ctx, int kmax, bool fp64) {
    int mx = 0;
    GGF_CK(cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    const int r = ctx->g.r, KRM = kmax * r;
    const size_t cw = fp64 ? sizeof(cxd) : sizeof(cxf);
    const size_t need_apply = apply_smem(2, KRM, cw) + 1024;
    if (!ggf_steps_fit(ctx, kmax, fp64) || need_apply > (size_t)mx)
        return ggf_fail(ctx, GGF_EINVAL, "delay too large: batch kernels need more shared memory than the device has");
    return GGF_OK;
}

// Run links l0 .. l0 + kb - 1 of the sweep as one batch (gather, link steps,
// X applied to the V panel, flush).
ggf_status ggf_batch(ggf_ctx* ctx, int l0, int kb, cudaStream_t st) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    const bool fp64 = ch.opts.precision == GGF_FP64;
    const int N = g.N, r = g.r, KRM = ch.kmax * r, kr = kb * r;
    const size_t rsz = fp64 ? sizeof(double) : sizeof(float);
    const size_t ssz = (size_t)ch.n * 2 * KRM * KRM * rsz;   // one family pair's small matrices, all chains
    void* Sr = ch.Sm;
    void* Sc_ = (unsigned char*)ch.Sm + ssz * ctx->K;
    const int ev0 = ctx->prof_mark(st);
    {
        const int br_r = gather_rows(kr, rsz), br_c = gather_rows(kr, 2 * rsz);
        dim3 gr((N + br_r - 1) / br_r, ctx->K, ch.n), gc((N + br_c - 1) / br_c, ctx->Kc, ch.n);
        const size_t t0 = (kr * sizeof(int) + 15) & ~(size_t)15;
        if (fp64) {
            batch_gather<double><<<gr, 256, t0 + (size_t)br_r * (kr + 1) * rsz, st>>>(
                g, l0, kb, ctx->K, KRM, br_r, (const double*)ch.Wr, (double*)ch.Pr, (double*)Sr);
            if (ctx->Kc)
                batch_gather<cxd><<<gc, 256, t0 + (size_t)br_c * (kr + 1) * 2 * rsz, st>>>(
                    g, l0, kb, ctx->Kc, KRM, br_c, (const cxd*)ch.Wc, (double*)ch.Pc, (cxd*)Sc_);
        } else {
            batch_gather<float><<<gr, 256, t0 + (size_t)br_r * (kr + 1) * rsz, st>>>(
                g, l0, kb, ctx->K, KRM, br_r, (const float*)ch.Wr, (float*)ch.Pr, (float*)Sr);
            if (ctx->Kc)
                batch_gather<cxf><<<gc, 256, t0 + (size_t)br_c * (kr + 1) * 2 * rsz, st>>>(
                    g, l0, kb, ctx->Kc, KRM, br_c, (const cxf*)ch.Wc, (float*)ch.Pc, (cxf*)Sc_);
        }
        GGF_CK(cudaGetLastError());
    }
    const int ev1 = ctx->prof_mark(st);
    ctx->prof_pair(GGF_KT_GATHER, ev0, ev1);
    GGF_TRY(ggf_batch_steps(ctx, l0, kb, Sr, Sc_, st));
    const int ev2 = ctx->prof_mark(st);
    ctx->prof_pair(GGF_KT_RATIO, ev1, ev2);
    {
        int mx = 0;
        GGF_CK(cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
        // 64-row blocks where they fit in shared memory, else 32
        const int rpt_r = apply_smem(4, kr, rsz) + 1024 <= (size_t)mx ? 4 : 2;
        const int rpt_c = apply_smem(4, kr, 2 * rsz) + 1024 <= (size_t)mx ? 4 : 2;
        dim3 gr((N + 16 * rpt_r - 1) / (16 * rpt_r), ctx->K, ch.n), gc((N + 16 * rpt_c - 1) / (16 * rpt_c), ctx->Kc, ch.n);
        const size_t sr = apply_smem(rpt_r, kr, rsz), sc = apply_smem(rpt_c, kr, 2 * rsz);
#define GGF_APPLY(T, RPT, grid, smem, fam, Pp, Sp) \
    batch_apply<T, RPT><<<grid, 256, smem, st>>>(N, fam, KRM, kr, (typename Sc<T>::R*)(Pp), (const T*)(Sp), ch.pend)
        if (GGF_APPLY_TC && !fp64 && ctx->use_tc && kr <= 256 && g.group != GGF_Z2) {
            // FP32 chains: the X product on the tensor cores (TF32 split).  Z2
            // chains keep the FMA-pipe product: a flip is a large change, and
            // the tensor-core accumulation doubled their FP32 drift (measured
            // 3.3e-6 against 1.7e-6 per accept at 16 x 16), while the small
            // moves of U(1) and SU(2) chains are unaffected (1e-8 per accept)
            GGF_TRY(ggf_apply_tc(ctx, false, ctx->K, kr, (float*)ch.Pr, (const float*)Sr, st));
            GGF_TRY(ggf_apply_tc(ctx, true, ctx->Kc, kr, (float*)ch.Pc, (const float*)Sc_, st));
        } else if (fp64) {
            if (rpt_r == 4) GGF_APPLY(double, 4, gr, sr, ctx->K, ch.Pr, Sr); else GGF_APPLY(double, 2, gr, sr, ctx->K, ch.Pr, Sr);
            if (ctx->Kc) {
                if (rpt_c == 4) GGF_APPLY(cxd, 4, gc, sc, ctx->Kc, ch.Pc, Sc_); else GGF_APPLY(cxd, 2, gc, sc, ctx->Kc, ch.Pc, Sc_);
            }
        } else {
            if (rpt_r == 4) GGF_APPLY(float, 4, gr, sr, ctx->K, ch.Pr, Sr); else GGF_APPLY(float, 2, gr, sr, ctx->K, ch.Pr, Sr);
            if (ctx->Kc) {
                if (rpt_c == 4) GGF_APPLY(cxf, 4, gc, sc, ctx->Kc, ch.Pc, Sc_); else GGF_APPLY(cxf, 2, gc, sc, ctx->Kc, ch.Pc, Sc_);
            }
        }
#undef GGF_APPLY
        GGF_CK(cudaGetLastError());
    }
    ctx->prof_pair(GGF_KT_APPLY, ev2, ctx->prof_mark(st));
    ctx->launches += 1 + 2 * (1 + (ctx->Kc ? 1 : 0));
    ch.steps_since_flush = kb;
    return ggf_flush(ctx, st);
}
