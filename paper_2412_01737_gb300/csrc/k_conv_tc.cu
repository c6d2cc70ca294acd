// The proposal network's 3 x 3 circular convolutions as implicit GEMMs on the
// sm_103a tensor cores (tcgen05.mma, accumulators in TMEM).
//
//   forward      Y[b][o][s] = bias[o] + sum_{t, c} W[o][c][t] X[b][c][nb_t(s)]
//                D[s][o] (M = pixels, N = output channels, K = taps x input
//                channels), BF16 operands (kind::f16), FP32 accumulation;
//   input grad   dX[b][c][s] = [act > 0] sum_{t, o} W[o][c][t] dY[b][o][nb'_t(s)]
//                D[s][c] (K = taps x output channels), TF32 operands
//                (kind::tf32: dY is FP32, rounded to TF32 once);
//   weight grad  dW[o][c][t] = sum_{b, s} X[b][c][nb_t(s)] dY[b][o][s]
//                D[(t, c)][o] (K = pixels of the CTA's bands), TF32, a plane
//                of partial sums per CTA, added up in a fixed order.
// nb_t(s) is pixel s shifted by tap t = 3 ky + kx, (ky - 1, kx - 1), on the
// torus; nb'_t(s) the opposite shift (the output pixel whose tap t read s).
//
// One CTA of 256 threads.  Forward and input gradient: every thread builds one
// row of the im2col operand tile per K step from values it loaded two steps
// earlier (the gather from global memory, which stays in L2), one thread issues
// the MMAs, and two operand buffers alternate.  The weight operand lies in global
// memory in the shared-memory layout already (ggf_conv_pack.cuh, kept up to date by
// the optimiser step), so that it is a plain copy.  Weight gradient: a
// band of rows of one sample is staged in shared memory, the inputs with their
// halo, and the tiles are built from there.  Mbarrier waits are bounded; on expiry the CTA stops,
// raises the network's error word and frees its TMEM.
//
// What bounds them: the operand building (index arithmetic and load latency),
// far above the MMAs.  Per layer 64 -> 64 at 16 x 16 and 128 samples, against
// gathering at the step of use, integer divisions per element and weights
// gathered by every CTA: forward 56 -> 40 us, input gradient 106 -> 61, weight
// gradient 221 -> 96 with the sum of its planes.
#include <cuda_bf16.h>
#include "ggf_ctx.h"
#include "ggf_tc.cuh"
#include "ggf_conv_pack.cuh"

namespace {

typedef __nv_bfloat16 bf16;
constexpr int CT = 256;                 // threads per CTA = im2col rows built per K step

__device__ __forceinline__ unsigned char* align1k(unsigned char* p) {
    return (unsigned char*)(((uintptr_t)p + 1023) & ~(uintptr_t)1023);
}

// pixel (x, y) shifted by sign * (kx, ky) of tap t on the torus
__device__ __forceinline__ int shifted(int L, int x, int y, int t, int sign) {
    int xx = x + sign * (t % 3 - 1), yy = y + sign * (t / 3 - 1);
    xx = xx < 0 ? xx + L : xx >= L ? xx - L : xx;
    yy = yy < 0 ? yy + L : yy >= L ? yy - L : yy;
    return yy * L + xx;
}

// 16-byte copy of a packed operand
__device__ __forceinline__ void copy_packed(unsigned char* dst, const void* src, int bytes) {
    const uint4* g = (const uint4*)src;
#pragma unroll 6
    for (int e = threadIdx.x; e < bytes / 16; e += CT) ((uint4*)dst)[e] = g[e];
}

// TMEM allocation by one whole warp; the column address lands in *slot
__device__ __forceinline__ void tmem_alloc_warp(uint32_t* slot, int ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(slot)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

// Operand-buffer bookkeeping shared by the three kernels: before a buffer is
// rewritten, the MMAs that read it (one commit) must have completed.  Every
// thread tracks the same state and takes the same waits; the outcome is
// agreed with __syncthreads_or so that no thread leaves a loop alone.
struct Bufs {
    uint32_t bar[2];
    uint32_t phase[2] = {0u, 0u};
    bool pending[2] = {false, false};
    __device__ bool wait(int b) {
        bool ok = true;
        if (pending[b]) {
            ok = tc::mbar_wait(bar[b], phase[b]);
            phase[b] ^= 1u;
            pending[b] = false;
        }
        return !__syncthreads_or(!ok);
    }
    __device__ bool drain() { return wait(0) && wait(1); }
};

__device__ __forceinline__ void fence_to_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---------------------------------------------------------------------------
// forward: two M tiles of 128 pixels per pass, N = CO_PAD output channels
template <int CI_PAD, int CO_PAD, bool RELU, bool OUT_F32>
__global__ void __launch_bounds__(CT, 1)
conv_fwd_tc(int n, int L, int ci, int co, const bf16* X, const void* Wp, const float* bias, void* Y, int* err) {
    constexpr int KT = 9 * CI_PAD, KS = KT / 16;
    constexpr int TCOLS = 2 * CO_PAD < 32 ? 32 : 2 * CO_PAD;
    constexpr uint32_t SBO_B = (KT / 8) * 128;
    extern __shared__ unsigned char smraw[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tslot;
    unsigned char* Bs = align1k(smraw);                       // CO_PAD x KT, k = t * CI_PAD + c
    unsigned char* As = Bs + CO_PAD * KT * 2;                 // 2 buffers x 2 tiles x 128 rows x 32 B
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int V = L * L;
    copy_packed(Bs, Wp, CO_PAD * KT * 2);
    if (warp == 0) tmem_alloc_warp(&tslot, TCOLS);
    Bufs bf;
    bf.bar[0] = tc::smem_u32(&bars[0]);
    bf.bar[1] = tc::smem_u32(&bars[1]);
    if (tid == 0) {
        tc::mbar_init(bf.bar[0], 1);
        tc::mbar_init(bf.bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    fence_to_async();
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tbase = tslot;
    bool ok = true;
    for (int b = blockIdx.x; b < n && ok; b += gridDim.x) {
        const bf16* Xb = X + (size_t)b * ci * V;
        for (int p0 = 0; p0 < V && ok; p0 += 2 * 128) {
            const int s = p0 + tid, x = s % L, y = s / L;
            // the 16 input channels of step ks, loaded two steps ahead of their use
            auto fetch = [&](int ks, uint32_t (&pk)[8]) {
                const int t = ks / (CI_PAD / 16), c0 = (ks % (CI_PAD / 16)) * 16;
                const bf16* src = Xb + (s < V ? shifted(L, x, y, t, 1) : 0);
                uint16_t v[16];
#pragma unroll
                for (int h = 0; h < 16; ++h)
                    v[h] = (s < V && c0 + h < ci) ? __bfloat16_as_ushort(src[(size_t)(c0 + h) * V]) : (uint16_t)0;
#pragma unroll
                for (int h = 0; h < 8; ++h) pk[h] = (uint32_t)v[2 * h] | ((uint32_t)v[2 * h + 1] << 16);
            };
            auto step = [&](int ks, uint32_t (&pk)[8]) -> bool {
                const int buf = ks & 1;
                if (!bf.wait(buf)) return false;
                unsigned char* Ab = As + buf * 8192 + (tid >> 7) * 4096;
                const int r = tid & 127;
                *(uint4*)(Ab + tc::cm32(r, 0, 2)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                *(uint4*)(Ab + tc::cm32(r, 8, 2)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                if (ks + 2 < KS) fetch(ks + 2, pk);
                fence_to_async();
                __syncthreads();
                if (tid == 0) {
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint64_t bd = tc::desc(tc::smem_u32(Bs + ks * 256), 128, SBO_B);
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const uint64_t ad = tc::desc(tc::smem_u32(As + buf * 8192 + m * 4096), 128, 256);
                        tc::mma_bf16(tbase + m * CO_PAD, ad, bd, tc::idesc_bf16(128, CO_PAD), ks > 0 ? 1u : 0u);
                    }
                    tc::commit(bf.bar[buf]);
                }
                bf.pending[buf] = true;
                return true;
            };
            uint32_t pa[8], pb[8];
            fetch(0, pa);
            fetch(1, pb);
            for (int ks = 0; ks < KS && ok; ks += 2) {
                ok = step(ks, pa);
                if (ok && ks + 1 < KS) ok = step(ks + 1, pb);
            }
            if (!ok || !(ok = bf.drain())) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            // epilogue: warp -> TMEM lane quarter q of tile m
            const int q = warp & 3, m = warp >> 2;
            const int sp = p0 + m * 128 + q * 32 + lane;
#pragma unroll
            for (int j = 0; j < CO_PAD; j += 16) {
                float v[16];
                tc::ld16(tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)(m * CO_PAD + j), v);
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const int o = j + k;
                    if (o < co && sp < V) {
                        float a = v[k] + bias[o];
                        if (RELU) a = fmaxf(a, 0.f);
                        const size_t oi = ((size_t)b * co + o) * V + sp;
                        if (OUT_F32) ((float*)Y)[oi] = a;
                        else ((bf16*)Y)[oi] = __float2bfloat16(a);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncthreads();
        }
    }
    bf.drain();
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(TCOLS));
    }
    if (!ok && tid == 0) atomicExch(err, 1);
}

// ---------------------------------------------------------------------------
// input gradient: D[s][c], N = 64 input channels, K = 9 x CO_PAD (TF32 steps of 8)
template <int CO_PAD>
__global__ void __launch_bounds__(CT, 1)
conv_bwd_data_tc(int n, int L, int ci, int co, const void* Wp, const float* dY, const bf16* act, float* dX,
                 int* err) {
    constexpr int NC = 64, KT = 9 * CO_PAD, KS = KT / 8, TCOLS = 2 * NC;
    constexpr uint32_t SBO_B = (KT / 4) * 128;
    extern __shared__ unsigned char smraw[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tslot;
    unsigned char* Bs = align1k(smraw);                       // NC x KT floats, k = t * CO_PAD + o
    unsigned char* As = Bs + NC * KT * 4;                     // 2 buffers x 2 tiles x 128 rows x 32 B
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int V = L * L;
    copy_packed(Bs, Wp, NC * KT * 4);
    if (warp == 0) tmem_alloc_warp(&tslot, TCOLS);
    Bufs bf;
    bf.bar[0] = tc::smem_u32(&bars[0]);
    bf.bar[1] = tc::smem_u32(&bars[1]);
    if (tid == 0) {
        tc::mbar_init(bf.bar[0], 1);
        tc::mbar_init(bf.bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    fence_to_async();
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tbase = tslot;
    bool ok = true;
    for (int b = blockIdx.x; b < n && ok; b += gridDim.x) {
        const float* dYb = dY + (size_t)b * co * V;
        for (int p0 = 0; p0 < V && ok; p0 += 2 * 128) {
            const int s = p0 + tid, x = s % L, y = s / L;
            // the 8 output channels of step ks, loaded two steps ahead of their use
            auto fetch = [&](int ks, float (&v)[8]) {
                const int t = ks / (CO_PAD / 8), o0 = (ks % (CO_PAD / 8)) * 8;
                const float* src = dYb + (s < V ? shifted(L, x, y, t, -1) : 0);
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = (s < V && o0 + k < co) ? src[(size_t)(o0 + k) * V] : 0.f;
            };
            auto step = [&](int ks, float (&v)[8]) -> bool {
                const int buf = ks & 1;
                if (!bf.wait(buf)) return false;
                unsigned char* Ab = As + buf * 8192 + (tid >> 7) * 4096;
                const int r = tid & 127;
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = tc::tf32_rna(v[k]);
                *(float4*)(Ab + tc::cm32(r, 0, 4)) = make_float4(v[0], v[1], v[2], v[3]);
                *(float4*)(Ab + tc::cm32(r, 4, 4)) = make_float4(v[4], v[5], v[6], v[7]);
                if (ks + 2 < KS) fetch(ks + 2, v);
                fence_to_async();
                __syncthreads();
                if (tid == 0) {
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint64_t bd = tc::desc(tc::smem_u32(Bs + ks * 256), 128, SBO_B);
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const uint64_t ad = tc::desc(tc::smem_u32(As + buf * 8192 + m * 4096), 128, 256);
                        tc::mma_tf32(tbase + m * NC, ad, bd, tc::idesc_tf32(128, NC), ks > 0 ? 1u : 0u);
                    }
                    tc::commit(bf.bar[buf]);
                }
                bf.pending[buf] = true;
                return true;
            };
            float va[8], vb[8];
            fetch(0, va);
            fetch(1, vb);
            for (int ks = 0; ks < KS && ok; ks += 2) {
                ok = step(ks, va);
                if (ok && ks + 1 < KS) ok = step(ks + 1, vb);
            }
            if (!ok || !(ok = bf.drain())) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const int q = warp & 3, m = warp >> 2;
            const int sp = p0 + m * 128 + q * 32 + lane;
#pragma unroll
            for (int j = 0; j < NC; j += 16) {
                float v[16];
                tc::ld16(tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)(m * NC + j), v);
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const int c = j + k;
                    if (c < ci && sp < V) {
                        const size_t xi = ((size_t)b * ci + c) * V + sp;
                        dX[xi] = (act && !(__bfloat162float(act[xi]) > 0.f)) ? 0.f : v[k];
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncthreads();
        }
    }
    bf.drain();
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(TCOLS));
    }
    if (!ok && tid == 0) atomicExch(err, 1);
}

// ---------------------------------------------------------------------------
// weight gradient: D[(t, c)][o], MT tiles of 128 rows (t, c), N = CO_PAD,
// K = pixels (TF32 steps of 8); the CTA's partial sums go to its own plane of
// `part` ([o][t][c]: a warp's 32 rows are 32 consecutive words), which
// reduce_weight_grad adds up in a fixed order.  Adding them to the gradient
// atomically cost a sector per word and made the sums, and with them the
// optimiser's normalised steps, depend on the CTAs' timing.  Work unit: h rows
// of a sample.
struct BandLayout {
    int xs, ys;              // elements between channels of the staged X (with halo) and dY
    size_t x, y, base, total;
};
__host__ __device__ inline BandLayout band_layout(int L, int ci, int co, int h, size_t front) {
    BandLayout l;
    // an odd number of words between channels: neighbouring channels on other banks
    l.xs = (h + 2) * (L + 2);
    l.xs += l.xs & 1;
    if ((l.xs >> 1) % 2 == 0) l.xs += 2;
    l.ys = h * L + 8;
    l.ys |= 1;
    size_t o = front;
    auto take = [&](size_t& at, size_t bytes) { at = o; o = (o + bytes + 15) & ~(size_t)15; };
    take(l.x, (size_t)ci * l.xs * 2);
    take(l.y, (size_t)co * l.ys * 4);
    take(l.base, (size_t)(h * L + 8) * 2);
    l.total = o;
    return l;
}

template <int MT, int CO_PAD>
__global__ void __launch_bounds__(CT, 1)
conv_bwd_weight_tc(int n, int L, int ci, int co, int h, const bf16* X, const float* dY, float* part, int* err) {
    constexpr int TC_ = MT * CO_PAD <= 32 ? 32 : MT * CO_PAD <= 64 ? 64 : MT * CO_PAD <= 128 ? 128
                        : MT * CO_PAD <= 256 ? 256 : 512;
    constexpr int ABYTES = MT * 128 * 32;                     // one buffer of A
    constexpr int BBYTES = CO_PAD * 32;                       // one buffer of B
    extern __shared__ unsigned char smraw[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tslot;
    unsigned char* As = align1k(smraw);
    unsigned char* Bsm = As + 2 * ABYTES;
    const BandLayout lay = band_layout(L, ci, co, h, 2 * ABYTES + 2 * BBYTES);
    bf16* Xs = (bf16*)(As + lay.x);                           // [ci][xs]: rows y0 - 1 .. y0 + h, columns -1 .. L
    float* Ys = (float*)(As + lay.y);                         // [co][ys]: the band's pixels, TF32, zeros behind
    uint16_t* base = (uint16_t*)(As + lay.base);              // pixel -> its offset in a halo plane, less one row and column
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int V = L * L, R = 9 * ci, W2 = L + 2;              // rows (t, c) = t * ci + c
    if (warp == 0) tmem_alloc_warp(&tslot, TC_);
    Bufs bf;
    bf.bar[0] = tc::smem_u32(&bars[0]);
    bf.bar[1] = tc::smem_u32(&bars[1]);
    if (tid == 0) {
        tc::mbar_init(bf.bar[0], 1);
        tc::mbar_init(bf.bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    for (int q = tid; q < h * L + 8; q += CT) base[q] = (uint16_t)(q < h * L ? (q / L) * W2 + q % L : 0);
    // this thread's (t, c) rows: their offset in Xs, -1 past the last
    int off[MT];
#pragma unroll
    for (int i = 0; i < MT; ++i) {
        const int row = (tid + i * CT) >> 1, t = row / ci, c = row - t * ci;
        off[i] = row < R ? c * lay.xs + (t / 3) * W2 + t % 3 : -1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tbase = tslot;
    const int bands = (L + h - 1) / h;
    bool ok = true;
    int step = 0;
    for (int u = blockIdx.x; u < n * bands && ok; u += gridDim.x) {
        const int b = u / bands, y0 = (u - b * bands) * h, hh = min(h, L - y0), npx = hh * L;
        const bf16* Xb = X + (size_t)b * ci * V;
        const float* dYb = dY + (size_t)b * co * V + (size_t)y0 * L;
        // the staged band is not rewritten while its tiles are being built: the
        // last build ended with a barrier
        for (int rr = warp; rr < ci * (hh + 2); rr += CT / 32) {
            const int c = rr / (hh + 2), yy = rr - c * (hh + 2);
            int gy = y0 + yy - 1;
            gy = gy < 0 ? gy + L : gy >= L ? gy - L : gy;
            const bf16* src = Xb + (size_t)c * V + (size_t)gy * L;
            bf16* dst = Xs + (size_t)c * lay.xs + yy * W2;
            for (int x = lane; x < W2; x += 32) dst[x] = src[x == 0 ? L - 1 : x == L + 1 ? 0 : x - 1];
        }
        for (int o = warp; o < co; o += CT / 32) {
            for (int q = lane; q < ((npx + 7) & ~7); q += 32)
                Ys[(size_t)o * lay.ys + q] = q < npx ? tc::tf32_rna(dYb[(size_t)o * V + q]) : 0.f;
        }
        __syncthreads();
        for (int s0 = 0; s0 < npx && ok; s0 += 8, ++step) {
            const int buf = step & 1;
            if (!(ok = bf.wait(buf))) break;
            unsigned char* Ab = As + buf * ABYTES;
            // A: rows (t, c), 8 pixels; 4-wide groups of k per store.  Pixels past
            // the band meet zeros of dY, and read the band's first pixel (never
            // what shared memory held before)
            const int kg = (tid & 1) * 4;
            ushort4 q4 = *(const ushort4*)(base + s0 + kg);
            if (s0 + 8 > npx) {
                if (s0 + kg + 0 >= npx) q4.x = 0;
                if (s0 + kg + 1 >= npx) q4.y = 0;
                if (s0 + kg + 2 >= npx) q4.z = 0;
                if (s0 + kg + 3 >= npx) q4.w = 0;
            }
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                const int row = (tid + i * CT) >> 1;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (off[i] >= 0) {
                    const bf16* p = Xs + off[i];
                    v = make_float4(__bfloat162float(p[q4.x]), __bfloat162float(p[q4.y]), __bfloat162float(p[q4.z]),
                                    __bfloat162float(p[q4.w]));
                }
                *(float4*)(Ab + (row >> 7) * 4096 + tc::cm32(row & 127, kg, 4)) = v;
            }
            unsigned char* Bb = Bsm + buf * BBYTES;
            if (tid < CO_PAD * 2) {
                const int o = tid >> 1;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (o < co) {
                    const float* p = Ys + (size_t)o * lay.ys + s0 + kg;
                    v = make_float4(p[0], p[1], p[2], p[3]);
                }
                *(float4*)(Bb + tc::cm32(o, kg, 4)) = v;
            }
            fence_to_async();
            __syncthreads();
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint64_t bd = tc::desc(tc::smem_u32(Bb), 128, 256);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const uint64_t ad = tc::desc(tc::smem_u32(Ab + m * 4096), 128, 256);
                    tc::mma_tf32(tbase + m * CO_PAD, ad, bd, tc::idesc_tf32(128, CO_PAD), step > 0 ? 1u : 0u);
                }
                tc::commit(bf.bar[buf]);
            }
            bf.pending[buf] = true;
        }
    }
    if (ok) ok = bf.drain();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok && step > 0) {
        // warp -> lane quarter q; the tiles are shared out over the two warp halves
        const int q = warp & 3;
        for (int m = warp >> 2; m < MT; m += 2) {
            const int row = m * 128 + q * 32 + lane;
#pragma unroll
            for (int j = 0; j < CO_PAD; j += 16) {
                float v[16];
                tc::ld16(tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)(m * CO_PAD + j), v);
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const int o = j + k;
                    if (o < co && row < R) part[((size_t)blockIdx.x * co + o) * R + row] = v[k];
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(TC_));
    }
    if (!ok && tid == 0) atomicExch(err, 1);
}

// dW [o][c][t] = sum of the planes of part [o][t][c]: eight threads per word,
// each over every eighth plane, then a tree.
__global__ void __launch_bounds__(256) reduce_weight_grad(int planes, int ci, int co, const float* part, float* dW) {
    __shared__ float red[8][33];
    const int R = 9 * ci, e = blockIdx.x * 32 + (threadIdx.x & 31), g = threadIdx.x >> 5;
    float acc = 0.f;
    if (e < co * R)
#pragma unroll 4
        for (int k = g; k < planes; k += 8) acc += part[(size_t)k * co * R + e];
    red[g][threadIdx.x & 31] = acc;
    __syncthreads();
    if (g == 0 && e < co * R) {
        const int x = threadIdx.x & 31, o = e / R, t = (e - o * R) / ci, c = e % ci;
        dW[((size_t)o * ci + c) * 9 + t] = ((red[0][x] + red[1][x]) + (red[2][x] + red[3][x])) +
                                           ((red[4][x] + red[5][x]) + (red[6][x] + red[7][x]));
    }
}

// db[o] = sum_{b, s} dY[b][o][s].  A thread's values are added one after the
// other (the sums cancel to a fraction of their terms, and the optimiser
// normalises them, so that another order shows), but loaded eight at a time.
__global__ void conv_bias_grad(int n, int V, int co, const float* dY, float* db) {
    const int o = blockIdx.x, total = n * V;
    float acc = 0.f;
    int b = threadIdx.x / V, s = threadIdx.x - b * V;
    for (int e = threadIdx.x; e < total; e += 8 * blockDim.x) {
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[k] = e + k * (int)blockDim.x < total ? dY[((size_t)b * co + o) * V + s] : 0.f;
            s += blockDim.x;
            while (s >= V) { s -= V; ++b; }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (e + k * (int)blockDim.x < total) acc += v[k];
    }
    __shared__ float red[32];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float v = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
        db[o] = v;
    }
}

}  // namespace

// Dynamic shared memory of a launch: at least what the kernel uses, and at
// least enough that the CTAs resident on one SM never ask for more than the
// 512 TMEM columns together (a tcgen05.alloc beyond them would wait for a
// neighbour to finish): 60 KB (at most three CTAs) for up to 128 columns,
// 120 KB (one CTA) for 512.
static size_t launch_smem(size_t need, int tmem_cols) {
    const size_t floor_ = tmem_cols > 128 ? (size_t)120 << 10 : (size_t)60 << 10;
    return need > floor_ ? need : floor_;
}

// Host launchers (the kernels stride over samples; grid at most one CTA per
// SM).  ci, co: the layer's real channel counts (8 -> 64 -> 64 -> 64 -> 6).
ggf_status ggf_conv_fwd_tc(int n, int L, int ci, int co, bool relu, const void* X, const void* W, const float* bias,
                           void* Y, bool out_f32, int* err, int sms, cudaStream_t st) {
    const int grid = n < sms ? n : sms;
    if (grid == 0) return GGF_OK;
    cudaError_t e = cudaSuccess;
#define GGF_FWD(CIP, COP, RL, OF)                                                                              \
    do {                                                                                                       \
        const size_t sm = launch_smem(1024 + (size_t)(COP) * 9 * (CIP) * 2 + 2 * 8192, 2 * (COP));            \
        e = cudaFuncSetAttribute(conv_fwd_tc<CIP, COP, RL, OF>, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                                 (int)sm);                                                                     \
        if (e == cudaSuccess)                                                                                  \
            conv_fwd_tc<CIP, COP, RL, OF><<<grid, CT, sm, st>>>(n, L, ci, co, (const bf16*)X, W, bias, Y, err);                                 \
    } while (0)
    if (ci <= 16 && co <= 64 && relu && !out_f32) GGF_FWD(16, 64, true, false);
    else if (ci <= 64 && co <= 64 && co > 16 && relu && !out_f32) GGF_FWD(64, 64, true, false);
    else if (ci <= 64 && co <= 16 && !relu && out_f32) GGF_FWD(64, 16, false, true);
    else return GGF_EINVAL;
#undef GGF_FWD
    if (e != cudaSuccess) return GGF_ECUDA;
    return cudaGetLastError() == cudaSuccess ? GGF_OK : GGF_ECUDA;
}

ggf_status ggf_conv_bwd_data_tc(int n, int L, int ci, int co, const void* W, const float* dY, const void* act,
                                float* dX, int* err, int sms, cudaStream_t st) {
    const int grid = n < sms ? n : sms;
    if (grid == 0) return GGF_OK;
    if (ci > 64) return GGF_EINVAL;
    cudaError_t e = cudaSuccess;
#define GGF_BWD(COP)                                                                                           \
    do {                                                                                                       \
        const size_t sm = launch_smem(1024 + (size_t)64 * 9 * (COP) * 4 + 2 * 8192, 128);                     \
        e = cudaFuncSetAttribute(conv_bwd_data_tc<COP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm); \
        if (e == cudaSuccess)                                                                                  \
            conv_bwd_data_tc<COP><<<grid, CT, sm, st>>>(n, L, ci, co, W, dY, (const bf16*)act, dX, err);                                              \
    } while (0)
    if (co <= 8) GGF_BWD(8);
    else if (co <= 64) GGF_BWD(64);
    else return GGF_EINVAL;
#undef GGF_BWD
    if (e != cudaSuccess) return GGF_ECUDA;
    return cudaGetLastError() == cudaSuccess ? GGF_OK : GGF_ECUDA;
}

// part: scratch of sms co 9 ci floats.  A unit of work is the
// tallest band of rows that fits in shared memory, or a shorter one where the
// samples alone would leave SMs idle.
ggf_status ggf_conv_bwd_weight_tc(int n, int L, int ci, int co, const void* X, const float* dY, float* dW,
                                  float* db, float* part, int* err, int sms, cudaStream_t st) {
    if (n < 1) return GGF_OK;
    cudaError_t e = cudaSuccess;
    int planes = 0;
    constexpr size_t cap = 227 * 1024 - 2048;
#define GGF_BWW(MT, COP)                                                                                              \
    do {                                                                                                              \
        const size_t front = 2 * ((size_t)(MT) * 128 * 32 + (size_t)(COP) * 32);                                      \
        int h = L;                                                                                                    \
        while (h > 1 && band_layout(L, ci, co, h, front).total > cap) --h;                                            \
        while (h > 2 && (long long)n * ((L + h - 1) / h) * 2 <= sms) h = (h + 1) / 2;                                  \
        const int units = n * ((L + h - 1) / h), grid = units < sms ? units : sms;                                     \
        planes = grid;                                                                                                \
        const size_t sm = launch_smem(1024 + band_layout(L, ci, co, h, front).total, (MT) * (COP));                    \
        e = cudaFuncSetAttribute(conv_bwd_weight_tc<MT, COP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm); \
        if (e == cudaSuccess)                                                                                         \
            conv_bwd_weight_tc<MT, COP><<<grid, CT, sm, st>>>(n, L, ci, co, h, (const bf16*)X, dY, part, err);         \
    } while (0)
    const int rows = 9 * ci;
    if (rows <= 128 && co <= 64) GGF_BWW(1, 64);
    else if (rows <= 640 && co <= 16) GGF_BWW(5, 16);
    else if (rows <= 640 && co <= 64) GGF_BWW(5, 64);
    else return GGF_EINVAL;
#undef GGF_BWW
    if (e != cudaSuccess) return GGF_ECUDA;
    reduce_weight_grad<<<(co * rows + 31) / 32, 256, 0, st>>>(planes, ci, co, part, dW);
    conv_bias_grad<<<co, 256, 0, st>>>(n, L * L, co, dY, db);
    return cudaGetLastError() == cudaSuccess ? GGF_OK : GGF_ECUDA;
}
