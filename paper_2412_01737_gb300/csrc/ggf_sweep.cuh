// Warp-level helpers and per-link pieces of a Metropolis link step, shared by
// the one-link-per-launch kernels (k_sample.cu) and the batched link steps
// on the small matrix W[T, T] (k_steps.cu).
#pragma once
#include <algorithm>
#include "ggf_ctx.h"
#include "ggf_geom.cuh"

namespace {
constexpr int NWARP = 8;
constexpr int MAXP = 36;           // pairs at K = 8
constexpr int MAXCS = 8;           // portable cluster size

// How a chain's pairs are dealt to the CTAs of its cluster: pairs
// ord[first[b]] .. ord[first[b + 1] - 1] belong to CTA b, real ones first.
struct PairBins {
    unsigned char first[MAXCS + 1], ord[MAXP];
};

// Bins of about one complex or two real pairs (a complex pair costs four real
// ones), at most MAXCS, the heaviest dealt first to the lightest bin.  Returns
// the number of CTAs.
inline int deal_pairs(int K, int Kc, PairBins& a) {
    const int P = K + Kc;
    const int CS = std::max(1, std::min(MAXCS, Kc + (K + 1) / 2));
    int load[MAXCS] = {0}, bin[MAXP], n = 0;
    for (int k = 0; k < P; ++k) {
        const int p = k < Kc ? K + k : k - Kc;       // complex pairs first
        int b = 0;
        for (int q = 1; q < CS; ++q)
            if (load[q] < load[b]) b = q;
        bin[p] = b;
        load[b] += p >= K ? 4 : 1;
    }
    for (int b = 0; b < CS; ++b) {
        a.first[b] = (unsigned char)n;
        for (int p = 0; p < P; ++p)
            if (bin[p] == b) a.ord[n++] = (unsigned char)p;
    }
    a.first[CS] = (unsigned char)n;
    return CS;
}

__device__ __forceinline__ double magc(cxd v) { return fabs(v.x) + fabs(v.y); }

// ---- FP64 scalars of the link steps: double for the diagonal pairs, cxd for
// the pairs n < m ----
__device__ __forceinline__ double magc(double v) { return fabs(v); }
// (on the words: an FP64 comparison takes the unit's 64 cycles too)
__device__ __forceinline__ bool is_zero(double v) { return ((__double2hiint(v) << 1) | __double2loint(v)) == 0; }
__device__ __forceinline__ bool is_zero(cxd v) { return is_zero(v.x) && is_zero(v.y); }
__device__ __forceinline__ bool is_fin(double v) { return isfinite(v); }
__device__ __forceinline__ bool is_fin(cxd v) { return isfinite(v.x) && isfinite(v.y); }
__device__ __forceinline__ double recip(double v) { return 1.0 / v; }
// one division where |v|^2 is well inside the range, Smith's method elsewhere
__device__ __forceinline__ cxd recip(cxd v) {
    const double m = v.x * v.x + v.y * v.y;
    const int e = __double2hiint(m) >> 20;          // biased exponent: 2^-930 <= m < 2^930
    if (e >= 1023 - 930 && e < 1023 + 930) {
        const double t = 1.0 / m;
        return {v.x * t, -v.y * t};
    }
    return cxd{1.0, 0.0} / v;
}
__device__ __forceinline__ void fmac(double& r, double a, double b) { r = fma(a, b, r); }
__device__ __forceinline__ void fmac(cxd& r, cxd a, cxd b) {
    r.x = fma(a.x, b.x, r.x); r.x = fma(-a.y, b.y, r.x);
    r.y = fma(a.x, b.y, r.y); r.y = fma(a.y, b.x, r.y);
}
__device__ __forceinline__ void fmsc(double& r, double a, double b) { r = fma(-a, b, r); }
__device__ __forceinline__ void fmsc(cxd& r, cxd a, cxd b) {
    r.x = fma(-a.x, b.x, r.x); r.x = fma(a.y, b.y, r.x);
    r.y = fma(-a.x, b.y, r.y); r.y = fma(-a.y, b.x, r.y);
}
// a / d from id ~ 1 / d: the quotient a id, corrected once by its remainder
__device__ __forceinline__ double quotient(double a, double d, double id) {
    const double q = a * id;
    return fma(fma(-q, d, a), id, q);
}
__device__ __forceinline__ cxd quotient(cxd a, cxd d, cxd id) {
    cxd q = a * id, r = a;
    fmsc(r, q, d);
    fmac(q, r, id);
    return q;
}
// The arithmetic of Z = (1 + Delta W_SS)^{-1} Delta.  Z of an FP32 chain is
// rounded to FP32, and one of some ten million elements lies so near the middle
// of two FP32 numbers that the last FP64 bits decide it; the chain then carries
// an FP32 rounding more or less.  So these chains keep one way of rounding
// (APART: the product first, then the sum; the quotient from a division);
// FP64 chains take fused sums and one reciprocal per row.
template <bool APART> struct ZOps {
    template <class T> __device__ static void add(T& r, T a, T b) { fmac(r, a, b); }
    template <class T> __device__ static void sub(T& r, T a, T b) { fmsc(r, a, b); }
    template <class T> __device__ static T inv(T d) { return recip(d); }
    template <class T> __device__ static T div(T a, T d, T id) { return quotient(a, d, id); }
};
template <> struct ZOps<true> {
    __device__ static double mul(double a, double b) { return __dmul_rn(a, b); }
    __device__ static cxd mul(cxd a, cxd b) {
        return {__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(a.y, b.x, __dmul_rn(a.x, b.y))};
    }
    __device__ static void add(double& r, double a, double b) { r = __dadd_rn(r, mul(a, b)); }
    __device__ static void sub(double& r, double a, double b) { r = __dsub_rn(r, mul(a, b)); }
    __device__ static void add(cxd& r, cxd a, cxd b) { const cxd t = mul(a, b); r = {__dadd_rn(r.x, t.x), __dadd_rn(r.y, t.y)}; }
    __device__ static void sub(cxd& r, cxd a, cxd b) { const cxd t = mul(a, b); r = {__dsub_rn(r.x, t.x), __dsub_rn(r.y, t.y)}; }
    template <class T> __device__ static T inv(T d) { return d; }
    template <class T> __device__ static T div(T a, T d, T) { return a / d; }
};
__device__ __forceinline__ cxd to_c(double v) { return {v, 0.0}; }
__device__ __forceinline__ cxd to_c(cxd v) { return v; }

// acc + a b and acc - a b as the FP32 chains have always rounded them (the
// product first); FP64 as fused steps, half the instructions of a unit that
// issues two FMAs per clock and SM.
template <class T> __device__ __forceinline__ void acc_add(T& r, T a, T b) { r += a * b; }
template <> __device__ __forceinline__ void acc_add<double>(double& r, double a, double b) { fmac(r, a, b); }
template <> __device__ __forceinline__ void acc_add<cxd>(cxd& r, cxd a, cxd b) { fmac(r, a, b); }
template <class T> __device__ __forceinline__ void acc_sub(T& r, T a, T b) { r -= a * b; }
template <> __device__ __forceinline__ void acc_sub<double>(double& r, double a, double b) { fmsc(r, a, b); }
template <> __device__ __forceinline__ void acc_sub<cxd>(cxd& r, cxd a, cxd b) { fmsc(r, a, b); }

// Lane of the largest magnitude among the lanes that take part (ties: the
// lowest lane), one warp, all lanes call: a redux over the upper words of the
// FP64 magnitudes, and over the lower words where those tie, instead of five
// shuffle rounds of three words (the search was a third of an elimination
// step).  The result is the same in every lane, so that callers branch alike
// whatever the values (NaN magnitudes order above all others).
__device__ __forceinline__ int warp_pivot(double m, bool part) {
    const unsigned hi = part ? (unsigned)__double2hiint(m) & 0x7fffffffu : 0u;
    const unsigned top = __reduce_max_sync(0xffffffffu, hi);
    unsigned cand = __ballot_sync(0xffffffffu, part && hi == top);
    if (__popc(cand) > 1) {
        const bool in = (cand >> (threadIdx.x & 31)) & 1;
        const unsigned lo = in ? (unsigned)__double2loint(m) : 0u;
        const unsigned best = __reduce_max_sync(0xffffffffu, lo);
        cand = __ballot_sync(0xffffffffu, in && lo == best);
    }
    return __ffs(cand) - 1;
}

// Pfaffian of an n x n (n <= 16) antisymmetric matrix in shared memory, by one
// warp (skew Gaussian elimination with pivoting).  A is destroyed.  An FP32
// inverse is antisymmetric only to its rounding, and which of two mirrored
// entries is read shows in the ratio: the multipliers come from the columns
// below the pivot, as everywhere in this library.  The update itself is
// antisymmetric, so each product is formed once for both triangles (12
// instead of 16 FP64 instructions; the FP64 unit issues two lanes per clock
// and SM), in three rounds of the warp at most.  Pairs are counted from the
// last row, so that a lane's (row, column) offsets are the same at every step.
template <class T>
__device__ __forceinline__ T warp_pfaffian(T* A, int n) {
    const int lane = threadIdx.x & 31;
    int pi[3], pj[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        const int e = lane + 32 * t;
        int i = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)e)) * 0.5f);
        if (i * (i - 1) / 2 > e) --i;
        if ((i + 1) * i / 2 <= e) ++i;
        pi[t] = i;
        pj[t] = e - i * (i - 1) / 2;
    }
    T res = Sc<T>::one();
    for (int k = 0; k < n - 1; k += 2) {
        const int q = k + 1;
        const bool part = lane > k && lane < n;
        const int p = warp_pivot(part ? magc(A[lane * n + k]) : 0.0, part);
        if (p != q) {
            if (lane >= k && lane < n) {
                const T t = A[q * n + lane]; A[q * n + lane] = A[p * n + lane]; A[p * n + lane] = t;
            }
            __syncwarp();
            if (lane >= k && lane < n) {
                const T t = A[lane * n + q]; A[lane * n + q] = A[lane * n + p]; A[lane * n + p] = t;
            }
            __syncwarp();
            res = -res;
        }
        const T piv = A[q * n + k];
        if (is_zero(piv)) { __syncwarp(); return Sc<T>::zero(); }
        res = res * A[k * n + q];
        if (k + 2 >= n) break;
        const T ip = recip(piv);
        // multipliers l_i = A[i][k] / A[q][k], one per row, in column k
        // (column k is not read again)
        if (lane > q && lane < n) A[lane * n + k] = A[lane * n + k] * ip;
        __syncwarp();
        const int mm = n - k - 2, cnt = mm * (mm - 1) / 2;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            if (32 * t >= cnt) break;
            if (lane + 32 * t < cnt) {
                const int i = n - 1 - pi[t], j = n - 1 - pj[t];
                T u = A[i * n + k] * A[j * n + q];
                fmsc(u, A[i * n + q], A[j * n + k]);
                A[i * n + j] += u;
                A[j * n + i] -= u;
            }
        }
        __syncwarp();
    }
    __syncwarp();
    return res;
}

// Solve [A | B] (r x 2r, row-major, stride 2r) in place by Gauss-Jordan with
// partial pivoting; the right half becomes A^{-1} B (columns up to the pivot
// are not read again and keep their values).  fcol: r scratch.
template <bool APART, class T>
__device__ __forceinline__ bool warp_solve(T* A, int r, T* fcol) {
    const int lane = threadIdx.x & 31;
    const int w = 2 * r;
    for (int k = 0; k < r; ++k) {
        const bool part = lane >= k && lane < r;
        const int p = warp_pivot(part ? magc(A[lane * w + k]) : 0.0, part);
        if (p != k) {
            if (lane < w) { T t = A[k * w + lane]; A[k * w + lane] = A[p * w + lane]; A[p * w + lane] = t; }
            __syncwarp();
        }
        const T d = A[k * w + k];
        if (is_zero(d)) return false;
        const T id = ZOps<APART>::inv(d);
        __syncwarp();
        if (lane > k && lane < w) A[k * w + lane] = ZOps<APART>::div(A[k * w + lane], d, id);
        if (lane < r) fcol[lane] = A[lane * w + k];
        __syncwarp();
        const int cols = w - k - 1;
        for (int e = lane; e < r * cols; e += 32) {
            const int i = e / cols, j = k + 1 + e % cols;
            if (i != k) ZOps<APART>::sub(A[i * w + j], fcol[i], A[k * w + j]);
        }
        __syncwarp();
    }
    return true;
}

// Pending-update panels of one (chain, pair): U (N x KRM) followed by V^T
// (N x KRM), K-major (row index first, rank index contiguous); complex
// values are stored as a real plane followed by an imaginary plane, so a
// (chain, pair) block holds 2 (real) or 4 (complex) planes of N * KRM.
template <class T> struct PanelIO {
    typedef typename Sc<T>::R R;
    static constexpr int PLANES = Sc<T>::CPLX ? 2 : 1;
    __device__ static T ld(const R* p, size_t plane, size_t idx);
    __device__ static void st(R* p, size_t plane, size_t idx, T v);
};
template <> __device__ __forceinline__ double PanelIO<double>::ld(const double* p, size_t, size_t i) { return p[i]; }
template <> __device__ __forceinline__ float PanelIO<float>::ld(const float* p, size_t, size_t i) { return p[i]; }
template <> __device__ __forceinline__ cxd PanelIO<cxd>::ld(const double* p, size_t pl, size_t i) { return {p[i], p[pl + i]}; }
template <> __device__ __forceinline__ cxf PanelIO<cxf>::ld(const float* p, size_t pl, size_t i) { return {p[i], p[pl + i]}; }
template <> __device__ __forceinline__ void PanelIO<double>::st(double* p, size_t, size_t i, double v) { p[i] = v; }
template <> __device__ __forceinline__ void PanelIO<float>::st(float* p, size_t, size_t i, float v) { p[i] = v; }
template <> __device__ __forceinline__ void PanelIO<cxd>::st(double* p, size_t pl, size_t i, cxd v) { p[i] = v.x; p[pl + i] = v.y; }
template <> __device__ __forceinline__ void PanelIO<cxf>::st(float* p, size_t pl, size_t i, cxf v) { p[i] = v.x; p[pl + i] = v.y; }

// Majorana offsets of the two ends of link l = 2 s + d: the source end (+d
// end of site s, which carries the twist) and the target end (-d end of the
// neighbour t).  Majorana xi < h2 of the link is a0 + xi, the others b0 + xi - h2.
GGF_HD void link_ends(const Geometry& g, int l, int& a0, int& b0) {
    const int s = l >> 1, d = l & 1, x = s % g.L, y = s / g.L;
    const int t = d == 0 ? y * g.L + (x + 1) % g.L : ((y + 1) % g.L) * g.L + x;
    a0 = s * g.B + (2 * d + 1) * g.h2;
    b0 = t * g.B + (2 * d) * g.h2;
}
GGF_HD int link_majorana(const Geometry& g, int a0, int b0, int xi) {
    return xi < g.h2 ? a0 + xi : b0 + xi - g.h2;
}

// One proposal (Sec. 5.1): accept draw, old and new link value.
struct Proposal {
    double u_acc, g_old, g_new, th_old, th_new;
};

// Philox4x64-10 with counter (sweep, link, 0, 0) and key (seed, chain):
// word 0 -> u_accept, word 1 -> u_propose.  Z2 flips the link; U(1) moves
// theta by width (u - 1/2) and wraps into [0, 2 pi).
__device__ __forceinline__ Proposal draw_proposal(const Geometry& g, const void* links, int c, int l,
                                                  unsigned long long sweep, uint64_t seed, double width,
                                                  uint64_t coff = 0) {
    uint64_t ctr[4] = {(uint64_t)sweep, (uint64_t)l, 0, 0}, out[4];
    philox4x64_10(ctr, seed, coff + (uint64_t)c, out);
    Proposal q;
    q.u_acc = u53(out[0]);
    const double u_prop = u53(out[1]);
    if (g.group == GGF_Z2) {
        double gv = (double)((const int8_t*)links)[(size_t)c * g.n_links + l];
        q.g_old = gv; q.g_new = -gv; q.th_old = 0.0; q.th_new = 0.0;
    } else {
        double th = ((const double*)links)[(size_t)c * g.n_links + l];
        double tn = th + width * (u_prop - 0.5);
        if (tn >= GGF_TWO_PI) tn -= GGF_TWO_PI;
        else if (tn < 0.0) tn += GGF_TWO_PI;
        q.g_old = 1.0; q.g_new = 1.0; q.th_old = th; q.th_new = tn;
    }
    return q;
}

// SU(2) proposal (n_v = 2, one doublet per link end), thread-local: with
// Philox words (u_acc, u_prop, u_z, u_phi) of counter (sweep, l, 0, 0) and
// key (seed, chain), g -> r g with r = cos d + i sin d (n . sigma),
// d = width (u_prop - 1/2), n = (sqrt(1 - z^2) cos phi, sqrt(1 - z^2) sin phi, z),
// z = 2 u_z - 1, phi = 2 pi u_phi, renormalised to a unit quaternion.  r and
// r^dag are equally likely (a Haar-symmetric move).  Writes the new
// quaternion and the old and new doublet rotations; returns u_acc.
GGF_HD double draw_su2(const Geometry& g, const void* links, int c, int l,
                                           unsigned long long sweep, uint64_t seed, double width, double* qn,
                                           double* Rold, double* Rnew, uint64_t coff = 0) {
    uint64_t ctr[4] = {(uint64_t)sweep, (uint64_t)l, 0, 0}, out[4];
    philox4x64_10(ctr, seed, coff + (uint64_t)c, out);
    const double d = width * (u53(out[1]) - 0.5);
    const double z = 2.0 * u53(out[2]) - 1.0;
    const double rho = sqrt(fmax(0.0, 1.0 - z * z));
    const double ph = GGF_TWO_PI * u53(out[3]);
    double sd, cd, sp, cp;
    sincos(d, &sd, &cd);
    sincos(ph, &sp, &cp);
    const double r[4] = {cd, sd * rho * cp, sd * rho * sp, sd * z};
    const double* q = link_quat(g, links, c, l);
    double t[4];
    quat_mul(r, q, t);
    const double nrm = sqrt(t[0] * t[0] + t[1] * t[1] + t[2] * t[2] + t[3] * t[3]);
    for (int k = 0; k < 4; ++k) qn[k] = t[k] / nrm;
    doublet_rotation(q, Rold);
    doublet_rotation(qn, Rnew);
    return u53(out[0]);
}

template <class T> struct Fp64Of;
template <> struct Fp64Of<double> { typedef double Z; };
template <> struct Fp64Of<float> { typedef double Z; };
template <> struct Fp64Of<cxd> { typedef cxd Z; };
template <> struct Fp64Of<cxf> { typedef cxd Z; };

template <class T> __device__ __forceinline__ typename Fp64Of<T>::Z wide(T v);
template <> __device__ __forceinline__ double wide<double>(double v) { return v; }
template <> __device__ __forceinline__ double wide<float>(float v) { return v; }
template <> __device__ __forceinline__ cxd wide<cxd>(cxd v) { return v; }
template <> __device__ __forceinline__ cxd wide<cxf>(cxf v) { return {(double)v.x, (double)v.y}; }
__device__ __forceinline__ double narrow(double v, double) { return v; }
__device__ __forceinline__ float narrow(double v, float) { return (float)v; }
__device__ __forceinline__ cxd narrow(cxd v, cxd) { return v; }
__device__ __forceinline__ cxf narrow(cxd v, cxf) { return {(float)v.x, (float)v.y}; }

// Element (xi, yi) of Delta = O' G O'^T - O G O^T of link l for pair p of its family.
template <class Z>
__device__ __forceinline__ Z delta_elem(const DevConst& dc, int p, int l, int xi, int yi, const Proposal& q,
                                        const double* tw, bool su2) {
    if (su2) return twisted_su2<Z>(dc, p, l, xi, yi, tw + 20) - twisted_su2<Z>(dc, p, l, xi, yi, tw + 4);
    return twisted_tab<Z>(dc, p, l, xi, yi, q.g_new, tw + 4) - twisted_tab<Z>(dc, p, l, xi, yi, q.g_old, tw);
}

// Pf(M') / Pf(M) = Pf([[Delta, -1], [1, W_SS]]) (r/2 = 2 n_v even: no extra
// sign), one warp; Bw is 2r x 2r scratch.
template <class T>
__device__ __forceinline__ T bordered_ratio(const T* D, const T* Ws, T* Bw, int r) {
    const int lane = threadIdx.x & 31, n2 = 2 * r;
    // a non-finite block (an inverse that overflowed) gives ratio 0: the
    // proposal is rejected
    bool fin = true;
    for (int e = lane; e < r * r; e += 32) fin = fin && is_fin(Ws[e]) && is_fin(D[e]);
    if (!__all_sync(0xffffffffu, fin)) return Sc<T>::zero();
    for (int e = lane; e < n2 * n2; e += 32) {
        int i = e / n2, j = e % n2;
        T v = Sc<T>::zero();
        if (i < r && j < r) v = D[i * r + j];
        else if (i >= r && j >= r) v = Ws[(i - r) * r + (j - r)];
        else if (i < r && j == i + r) v = -Sc<T>::one();
        else if (i >= r && j == i - r) v = Sc<T>::one();
        Bw[e] = v;
    }
    __syncwarp();
    return warp_pfaffian(Bw, n2);
}

// Ordered Gaussian indices (n, m) of pair p: p < K is (p, p); the pairs n < m
// follow in lexicographic order.
GGF_HD void pair_nm(int K, int p, int& n, int& m) {
    if (p < K) { n = m = p; return; }
    int k = p - K;
    n = 0;
    while (k >= K - 1 - n) { k -= K - 1 - n; ++n; }
    m = n + 1 + k;
}

// Scale of the pair terms of one configuration: amax = max_p Re(logc_p + ell_p)
// and 1 / (N(G) e^{-amax}), N(G) = Re sum_p w_p e^{logc_p + ell_p}; then
// pair_norm gives N_nm(G) / N(G) for pair p (diagonal pairs real).
GGF_HD void pair_scale(const DevConst& dc, const cxd* ell_c, double& amax, double& iden) {
    amax = -INFINITY;
    for (int p = 0; p < dc.P; ++p) amax = fmax(amax, dc.logc[p].x + ell_c[p].x);
    double den = 0.0;
    for (int p = 0; p < dc.P; ++p) {
        cxd e = dc.logc[p] + ell_c[p];
        if (p < dc.K) e.y = 0.0;
        e.x -= amax;
        den += (dc.w[p] * cexp_(e)).x;
    }
    iden = 1.0 / den;
}
GGF_HD cxd pair_norm(const DevConst& dc, const cxd* ell_c, int p, double amax, double iden) {
    cxd e = dc.logc[p] + ell_c[p];
    if (p < dc.K) e.y = 0.0;
    e.x -= amax;
    return iden * cexp_(e);
}

// Z = (1 + Delta W_SS)^{-1} Delta (r x r) into Zout, one warp; Aug is r x 2r
// scratch, fcol r; APART for FP32 chains (ZOps).  Returns false for a singular system.
template <bool APART, class T, class Z>
__device__ __forceinline__ bool pair_z(const T* D, const T* Ws, T* Aug, T* fcol, int r, Z* Zout) {
    const int lane = threadIdx.x & 31, w2 = 2 * r;
    for (int e = lane; e < r * r; e += 32) {
        const int i = e / r, j = e % r;
        T v = i == j ? Sc<T>::one() : Sc<T>::zero();
        for (int z = 0; z < r; ++z) ZOps<APART>::add(v, D[i * r + z], Ws[z * r + j]);
        Aug[i * w2 + j] = v;
        Aug[i * w2 + r + j] = D[e];
    }
    __syncwarp();
    const bool ok = warp_solve<APART>(Aug, r, fcol);
    for (int e = lane; e < r * r; e += 32) {
        const T v = Aug[(e / r) * w2 + r + e % r];
        if constexpr (sizeof(Z) == sizeof(T)) Zout[e] = v;
        else Zout[e] = to_c(v);
    }
    __syncwarp();
    return ok;
}

// ell_p += log rho_p: modulus only for diagonal pairs, phase wrapped into
// (-pi, pi] for pairs n < m.
__device__ __forceinline__ void ell_add(cxd& el, cxd rho, bool real_pair) {
    if (real_pair) {
        el.x += log(fabs(rho.x));        // a real ratio
    } else {
        el = el + clog_(rho);
        if (el.y > M_PI) el.y -= 2 * M_PI;
        else if (el.y <= -M_PI) el.y += 2 * M_PI;
    }
}

}  // namespace
