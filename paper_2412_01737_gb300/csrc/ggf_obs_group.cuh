// Cooperative bodies of the observable kernels: a group of lanes (one per
// virtual Majorana of a site: B = 8 n_v) evaluates one (chain, item).  What
// each item is, and the one-thread form of the same arithmetic, is in
// ggf_obs.cuh.
//
// One thread per item walked its W block row by row: dependent scattered
// loads, the pair weights' exponentials formed again by every thread, complex
// arithmetic for the real pairs and both orders of a complex pair from
// scratch.  Here a lane owns a row of the block (whole 16-byte pieces of it),
// the weights are formed once per CTA, real pairs stay real, and the two
// orders of a pair share their products (below).
#pragma once
#include "ggf_obs.cuh"

namespace {

constexpr int OT = 128;                 // threads per CTA

template <class T> struct Wide;         // FP64 type of an element of W
template <> struct Wide<double> { typedef double Z; };
template <> struct Wide<float> { typedef double Z; };
template <> struct Wide<cxd> { typedef cxd Z; };
template <> struct Wide<cxf> { typedef cxd Z; };

__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) { return (double)v; }
__device__ __forceinline__ cxd widen(cxd v) { return v; }
__device__ __forceinline__ cxd widen(cxf v) { return {(double)v.x, (double)v.y}; }

__device__ __forceinline__ void axpy(double& r, double a, double b) { r = fma(a, b, r); }
__device__ __forceinline__ void axpy(cxd& r, double a, cxd b) { r.x = fma(a, b.x, r.x); r.y = fma(a, b.y, r.y); }
__device__ __forceinline__ void axpy(cxd& r, cxd a, cxd b) {
    r.x = fma(a.x, b.x, r.x); r.x = fma(-a.y, b.y, r.x);
    r.y = fma(a.x, b.y, r.y); r.y = fma(a.y, b.x, r.y);
}
__device__ __forceinline__ cxd as_cx(double v) { return {v, 0.0}; }
__device__ __forceinline__ cxd as_cx(cxd v) { return v; }
__device__ __forceinline__ double shfl_xor_(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ cxd shfl_xor_(cxd v, int o) {
    return {__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
}

// n consecutive elements of W (n sizeof(T) a multiple of 8; 16-byte pieces
// where the run allows: every run starts on a multiple of its length)
template <int n, class T>
__device__ __forceinline__ void load_run(const T* p, typename Wide<T>::Z* out) {
    constexpr int bytes = n * sizeof(T);
    if constexpr (bytes % 16 == 0) {
        union { float4 v[bytes / 16]; T t[n]; } u;
#pragma unroll
        for (int k = 0; k < bytes / 16; ++k) u.v[k] = ((const float4*)p)[k];
#pragma unroll
        for (int k = 0; k < n; ++k) out[k] = widen(u.t[k]);
    } else {
        union { float2 v[bytes / 8]; T t[n]; } u;
#pragma unroll
        for (int k = 0; k < bytes / 8; ++k) u.v[k] = ((const float2*)p)[k];
#pragma unroll
        for (int k = 0; k < n; ++k) out[k] = widen(u.t[k]);
    }
}

// N_nm(G) / N(G) of every pair of one chain into np (shared), by warp 0.
__device__ __forceinline__ void chain_weights(const DevConst& dc, const cxd* el, cxd* np) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        double amax = -INFINITY, den = 0.0;
        for (int p = lane; p < dc.P; p += 32) amax = fmax(amax, dc.logc[p].x + el[p].x);
        for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        for (int p = lane; p < dc.P; p += 32) {
            cxd e = dc.logc[p] + el[p];
            if (p < dc.K) e.y = 0.0;
            e.x -= amax;
            const cxd t = cexp_(e);
            np[p] = t;
            den += (dc.w[p] * t).x;
        }
        for (int o = 16; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
        const double iden = 1.0 / den;
        for (int p = lane; p < dc.P; p += 32) np[p] = iden * np[p];
    }
    __syncthreads();
}

// ---- electric ------------------------------------------------------------------
// With A the columns S of the block W[site, link] and G = W[site, link]
// Gamma_tw[link, S], the two orders of a pair are
//   X_f = U + i V,  X_r = conj(U - i V),  U = A_S - D_S G,  V = G_S + D_S A
// (D real): one product with Gamma_tw instead of two, and real for the
// diagonal pairs.
template <int H> struct ElectricShared {
    cxd gt[2 * H * H];          // Gamma_tw[link, S]
    cxd A[4 * H * H], G[4 * H * H];
    cxd U[H * H], V[H * H];
    double tw[16];
};

template <class T, int H, bool FIELD>
__device__ __forceinline__ cxd electric_pair(const DevConst& dc, int pf, int l, const T* W, int lane, double gval,
                                             ElectricShared<H>& sh) {
    typedef typename Wide<T>::Z Z;
    constexpr int R = 2 * H, B = 4 * H;
    const Geometry& g = dc.g;
    Z* gt = (Z*)sh.gt;
    Z* As = (Z*)sh.A;
    Z* Gs = (Z*)sh.G;
    int a0, b0;
    link_ends(g, l, a0, b0);
    const int s0 = (l >> 1) * g.B, loc0 = a0 - s0;
    for (int e = lane; e < R * H; e += B)
        gt[e] = g.group == GGF_SU2 ? twisted_su2<Z>(dc, pf, l, e / H, e % H, sh.tw)
                                   : twisted_tab<Z>(dc, pf, l, e / H, e % H, gval, sh.tw);
    Z w[R];
    const T* row = W + (size_t)(s0 + lane) * g.N;
    load_run<H>(row + a0, w);
    load_run<H>(row + b0, w + H);
    __syncwarp();
#pragma unroll
    for (int b = 0; b < H; ++b) {
        Z s = Sc<Z>::zero();
#pragma unroll
        for (int j = 0; j < R; ++j) axpy(s, w[j], gt[j * H + b]);
        As[lane * H + b] = w[b];
        Gs[lane * H + b] = s;
    }
    __syncwarp();
    if (lane < H * H) {
        const int a = lane / H, b = lane % H;
        const double* Dr = dc.D + ((size_t)(l >> 1) * B + loc0 + a) * B;
        Z u = As[(loc0 + a) * H + b], v = Gs[(loc0 + a) * H + b];
#pragma unroll 4
        for (int i = 0; i < B; ++i) {
            const double d = Dr[i];
            axpy(u, -d, Gs[i * H + b]);
            axpy(v, d, As[i * H + b]);
        }
        sh.U[lane] = as_cx(u);
        sh.V[lane] = as_cx(v);
    }
    __syncwarp();
    // lane 0: the (n, m) order, lane 1: (m, n)
    cxd out = {0.0, 0.0};
    if (lane < 2) {
        const double sg = lane ? -1.0 : 1.0;
        cxd X[H][H];
#pragma unroll
        for (int a = 0; a < H; ++a)
#pragma unroll
            for (int b = 0; b < H; ++b) {
                const cxd u = sh.U[a * H + b], v = sh.V[a * H + b];
                // -(U + i V) or -conj(U - i V), plus i on the diagonal
                X[a][b] = {-(u.x - sg * v.y), -sg * (u.y + sg * v.x)};
                if (a == b) X[a][b].y += 1.0;
            }
        out = insertion<H, FIELD>(g, X);
    }
    __syncwarp();
    return out;
}

// ---- fermionic -------------------------------------------------------------------
// X[alpha][beta] = B_s W[s, t] B_t^T; every lane of the group gets the result.
template <class T, int BW>
__device__ __forceinline__ void coupled_group(const DevConst& dc, const T* W, int s, int t, int lane,
                                              typename Wide<T>::Z (&X)[4]) {
    typedef typename Wide<T>::Z Z;
    const double* Bs = dc.Bp + (size_t)s * 2 * BW;
    const double* Bt = dc.Bp + (size_t)t * 2 * BW;
    Z w[BW], u0 = Sc<Z>::zero(), u1 = Sc<Z>::zero();
    load_run<BW>(W + (size_t)(s * BW + lane) * dc.g.N + (size_t)t * BW, w);
#pragma unroll
    for (int j = 0; j < BW; ++j) {
        axpy(u0, Bt[j], w[j]);
        axpy(u1, Bt[BW + j], w[j]);
    }
    const double b0 = Bs[lane], b1 = Bs[BW + lane];
    X[0] = b0 * u0; X[1] = b0 * u1; X[2] = b1 * u0; X[3] = b1 * u1;
#pragma unroll
    for (int o = BW / 2; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) X[k] = X[k] + shfl_xor_(X[k], o);
}

}  // namespace
