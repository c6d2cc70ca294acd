// The observable kernels' bodies (electric, Sec. 5.3; fermionic, Sec. 5.2; scores
// and per-pair norms): a group of lanes (one per virtual Majorana of a site:
// B = 8 n_v) evaluates one (chain, item).  Each body is cut into phases, what a
// lane does between two barriers; the kernels run the phases with a warp's
// lanes side by side, ggf_obs.cuh one lane after the other on the host, so
// that CPU tests check the kernels' own arithmetic and indices.
//
// One thread per item walked its W block row by row: dependent scattered
// loads, the pair weights' exponentials formed again by every thread, complex
// arithmetic for the real pairs and both orders of a complex pair from
// scratch.  Here a lane owns a row of the block (whole 16-byte pieces of it),
// the weights are formed once per CTA or, for many CTAs, once per chain, real
// pairs stay real, and the two orders of a pair share their products (below).
// With many chains the FP64 unit is what is left, and it takes a warp's
// instruction at the same price whatever the number of its lanes.
#pragma once
#include "ggf_ctx.h"
#include "ggf_sweep.cuh"

namespace {

constexpr int OT = 128;                 // threads per CTA

template <class T> struct Wide;         // FP64 type of an element of W
template <> struct Wide<double> { typedef double Z; };
template <> struct Wide<float> { typedef double Z; };
template <> struct Wide<cxd> { typedef cxd Z; };
template <> struct Wide<cxf> { typedef cxd Z; };

GGF_HD double widen(double v) { return v; }
GGF_HD double widen(float v) { return (double)v; }
GGF_HD cxd widen(cxd v) { return v; }
GGF_HD cxd widen(cxf v) { return {(double)v.x, (double)v.y}; }

GGF_HD void axpy(double& r, double a, double b) { r = fma(a, b, r); }
GGF_HD void axpy(cxd& r, double a, cxd b) { r.x = fma(a, b.x, r.x); r.y = fma(a, b.y, r.y); }
GGF_HD void axpy(cxd& r, cxd a, cxd b) {
    r.x = fma(a.x, b.x, r.x); r.x = fma(-a.y, b.y, r.x);
    r.y = fma(a.x, b.y, r.y); r.y = fma(a.y, b.x, r.y);
}
GGF_HD cxd as_cx(double v) { return {v, 0.0}; }
GGF_HD cxd as_cx(cxd v) { return v; }
__device__ __forceinline__ double shfl_xor_(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ cxd shfl_xor_(cxd v, int o) {
    return {__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
}

// n consecutive elements of W (n sizeof(T) a multiple of 8; 16-byte pieces
// where the run allows: every run starts on a multiple of its length)
template <int n, class T>
GGF_HD void load_run(const T* p, typename Wide<T>::Z* out) {
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

// The weights of one chain's pairs: N_nm(G) / N(G), and w_p N_nm(G) / N(G).
struct PairWeights {
    cxd np[36], E[36];
};

// By G lanes (a power of two, P <= G or G = 32) of a warp whose lanes all call;
// np, E: [P], in any memory; nothing is stored where live is false.
__device__ __forceinline__ void warp_weights(const DevConst& dc, const cxd* el, int G, bool live, cxd* np, cxd* E) {
    const int lane = (threadIdx.x & 31) & (G - 1);
    double amax = -INFINITY, den = 0.0;
    for (int p = lane; p < dc.P; p += G) amax = fmax(amax, dc.logc[p].x + el[p].x);
    for (int o = G / 2; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    // (P <= 36: a lane has two pairs at most, the second one seldom)
    auto term = [&](int p) {
        cxd e = dc.logc[p] + el[p];
        if (p < dc.K) e.y = 0.0;
        e.x -= amax;
        const cxd t = cexp_(e);
        den += (dc.w[p] * t).x;
        return t;
    };
    cxd t0 = {0.0, 0.0}, t1 = {0.0, 0.0};
    if (lane < dc.P) t0 = term(lane);
    if (lane + G < dc.P) t1 = term(lane + G);
    for (int o = G / 2; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    const double iden = 1.0 / den;
    auto put = [&](int p, cxd t) {
        const cxd v = iden * t;
        np[p] = v;
        E[p] = dc.w[p] * v;
    };
    if (live && lane < dc.P) put(lane, t0);
    if (live && lane + G < dc.P) put(lane + G, t1);
}

// The weights of chain c into shared memory: from `ready` [n][2][P]
// (ggf_obs_weights), or formed by the CTA's first warp.
__device__ __forceinline__ void chain_weights(const DevConst& dc, int c, const cxd* ell, const cxd* ready,
                                              PairWeights& pw) {
    if (ready) {
        const cxd* r = ready + (size_t)c * 2 * dc.P;
        for (int p = threadIdx.x; p < dc.P; p += blockDim.x) {
            pw.np[p] = r[p];
            pw.E[p] = r[dc.P + p];
        }
    } else if (threadIdx.x < 32) {
        warp_weights(dc, ell + (size_t)c * dc.P, 32, true, pw.np, pw.E);
    }
    __syncthreads();
}

// ---- electric (the derivation is in k_electric.cu) ---------------------------

// Pfaffian of an H x H antisymmetric matrix (H = 2 n_v = 2 or 4), closed form.
template <int H>
GGF_HD cxd small_pf(const cxd (&A)[H][H]);
template <>
GGF_HD cxd small_pf<2>(const cxd (&A)[2][2]) { return A[0][1]; }
template <>
GGF_HD cxd small_pf<4>(const cxd (&A)[4][4]) {
    return A[0][1] * A[2][3] - A[0][2] * A[1][3] + A[0][3] * A[1][2];
}

// Normalised expectation of the insertion from G = Gamma_O[S, S]; FIELD: the
// U(1) twist charge Q_l itself (the electric field) instead of Q_l^2.
template <int H, bool FIELD = false>
GGF_HD cxd insertion(const Geometry& g, const cxd (&G)[H][H]) {
    if constexpr (FIELD) {
        cxd val = {0.0, 0.0};
#pragma unroll
        for (int j = 0; j < H / 2; ++j) {
            cxd occ = G[2 * j][2 * j + 1];
            occ.x += 1.0;
            val += (0.5 * (double)g.q[j]) * occ;       // q_j <n_j>
        }
        return val;
    }
    if (g.group == GGF_Z2) {
        return (H / 2) % 2 ? -small_pf<H>(G) : small_pf<H>(G);    // (-1)^{n_v}
    }
    if constexpr (H == 4) {
        if (g.group == GGF_SU2) {
            // sum_a (Q^a)^2 on the doublet = (3/4)(n_0 + n_1 - 2 n_0 n_1)
            cxd o = G[0][1] + G[2][3];
            o.x += 2.0;                                  // 2 (<n_0> + <n_1>)
            cxd pr = G[0][1] + G[2][3] + small_pf<H>(G);
            pr.x += 1.0;                                 // 4 <n_0 n_1>
            return 0.375 * (o - pr);                     // (3/4)(o / 2 - 2 pr / 4)
        }
    }
    cxd val = {0.0, 0.0};
#pragma unroll
    for (int j = 0; j < H / 2; ++j) {
        const double qj = g.q[j];
        cxd occ = G[2 * j][2 * j + 1];
        occ.x += 1.0;
        val += (0.5 * qj * qj) * occ;
    }
    if constexpr (H == 4) {
        cxd pr = G[0][1] + G[2][3] + small_pf<H>(G);
        pr.x += 1.0;
        val += (0.5 * g.q[0] * g.q[1]) * pr;            // 2 q_0 q_1 <n_0 n_1>
    }
    return val;
}

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

// The twists of a link's modes (U(1): one per virtual mode, SU(2): the doublet's)
// into sh.tw, mode by mode, and the value of a Z2 link.
GGF_HD int electric_modes(const Geometry& g) { return g.group == GGF_SU2 ? 1 : g.group == GGF_U1 ? g.n_v : 0; }
template <int H>
GGF_HD void electric_twist(const Geometry& g, const void* links, int c, int l, int mode, ElectricShared<H>& sh) {
    if (g.group == GGF_SU2) {
        doublet_rotation(link_quat(g, links, c, l), sh.tw);
    } else {
        const double th = ((const double*)links)[(size_t)c * g.n_links + l];
        sincos(g.q[mode] * th, &sh.tw[2 * mode + 1], &sh.tw[2 * mode]);
    }
}
GGF_HD double electric_link(const Geometry& g, const void* links, int c, int l) {
    return g.group == GGF_Z2 ? (double)((const int8_t*)links)[(size_t)c * g.n_links + l] : 1.0;
}

// Phase 1: the lane's entries of Gamma_tw and its row of W[site, link] (a0, b0: the link's ends).
template <class T, int H>
GGF_HD void electric_load(const DevConst& dc, int pf, int l, int a0, int b0, const T* W, int lane, double gval,
                          ElectricShared<H>& sh, typename Wide<T>::Z (&w)[2 * H]) {
    typedef typename Wide<T>::Z Z;
    constexpr int R = 2 * H, B = 4 * H;
    const Geometry& g = dc.g;
    Z* gt = (Z*)sh.gt;
    for (int e = lane; e < R * H; e += B) {
        const int j = e / H, b = e % H;
        if (g.group == GGF_Z2) gt[e] = mulc((j < H ? gval : 1.0) * gval, bond_elem<Z>(dc, pf, l, j, b));
        else if (g.group == GGF_SU2) gt[e] = twisted_su2<Z>(dc, pf, l, j, b, sh.tw);
        else gt[e] = twisted_tab<Z>(dc, pf, l, j, b, gval, sh.tw);
    }
    const T* row = W + (size_t)((l >> 1) * B + lane) * g.N;
    load_run<H>(row + a0, w);
    load_run<H>(row + b0, w + H);
}

// Phase 2: the lane's row of A and G.
template <class T, int H>
GGF_HD void electric_rows(int lane, const typename Wide<T>::Z (&w)[2 * H], ElectricShared<H>& sh) {
    typedef typename Wide<T>::Z Z;
    const Z* gt = (const Z*)sh.gt;
    Z* As = (Z*)sh.A;
    Z* Gs = (Z*)sh.G;
#pragma unroll
    for (int b = 0; b < H; ++b) {
        Z s = Sc<Z>::zero();
#pragma unroll
        for (int j = 0; j < 2 * H; ++j) axpy(s, w[j], gt[j * H + b]);
        As[lane * H + b] = w[b];
        Gs[lane * H + b] = s;
    }
}

// Phase 3: an entry of U and of V per lane, or of one of them where the group
// has lanes for both (an FP64 instruction costs a warp the same whatever the
// number of its lanes).
template <class T, int H>
GGF_HD void electric_products(const DevConst& dc, int l, int a0, int lane, ElectricShared<H>& sh) {
    typedef typename Wide<T>::Z Z;
    constexpr int B = 4 * H, E = H * H;
    const Z* As = (const Z*)sh.A;
    const Z* Gs = (const Z*)sh.G;
    const int e = lane % E, a = e / H, b = e % H, at = a0 - (l >> 1) * B + a;
    const double* Dr = dc.D + ((size_t)(l >> 1) * B + at) * B;
    if constexpr (2 * E <= B) {
        const bool second = lane >= E;
        const Z* other = second ? As : Gs;
        Z s = second ? Gs[at * H + b] : As[at * H + b];
#pragma unroll 4
        for (int i = 0; i < B; ++i) axpy(s, second ? Dr[i] : -Dr[i], other[i * H + b]);
        (second ? (Z*)sh.V : (Z*)sh.U)[e] = s;
    } else {
        Z u = As[at * H + b], v = Gs[at * H + b];
#pragma unroll 4
        for (int i = 0; i < B; ++i) {
            const double d = Dr[i];
            axpy(u, -d, Gs[i * H + b]);
            axpy(v, d, As[i * H + b]);
        }
        ((Z*)sh.U)[e] = u;
        ((Z*)sh.V)[e] = v;
    }
}

// Phase 4: lane 0: the (n, m) order, lane 1: (m, n); a diagonal pair's orders are one.
template <class T, int H, bool FIELD>
GGF_HD cxd electric_value(const Geometry& g, int lane, const ElectricShared<H>& sh) {
    typedef typename Wide<T>::Z Z;
    if (lane >= (Sc<Z>::CPLX ? 2 : 1)) return {0.0, 0.0};
    const Z* U = (const Z*)sh.U;
    const Z* V = (const Z*)sh.V;
    cxd X[H][H];
#pragma unroll
    for (int a = 0; a < H; ++a)
#pragma unroll
        for (int b = 0; b < H; ++b) {
            // -(U + i V) or -conj(U - i V), plus i on the diagonal
            if constexpr (Sc<Z>::CPLX) {
                const double sg = lane ? -1.0 : 1.0;
                const cxd u = U[a * H + b], v = V[a * H + b];
                X[a][b] = {-(u.x - sg * v.y), -sg * (u.y + sg * v.x)};
            } else {
                X[a][b] = {-U[a * H + b], -V[a * H + b]};
            }
            if (a == b) X[a][b].y += 1.0;
        }
    return insertion<H, FIELD>(g, X);
}

// The lane's order of pair p (value v, norm Np, weight E) into its sum and the per-pair
// output po [K][K] (or null; not live: nothing is stored).  w_p = 2 lambda_n^* lambda_m: the (n, m) term
// (lane 0) takes E / 2, the (m, n) term (lane 1) its conjugate; a diagonal pair
// E once.
GGF_HD void electric_term(const DevConst& dc, int p, int lane, bool live, cxd Np, cxd E, cxd v, cxd& num,
                         cxd* po) {
    const int K = dc.K;
    const bool cplx = p >= K;
    if (!cplx) {
        if (lane == 0) num += E * v;
    } else if (lane < 2) {
        num += 0.5 * ((lane ? conjg(E) : E) * v);
    }
    if (po && live) {
        int n, m;
        pair_nm(K, p, n, m);
        if (lane == 0) po[n * K + m] = Np * v;
        else if (lane == 1 && cplx) po[m * K + n] = conjg(Np) * v;
    }
}

template <class T, int H, bool FIELD>
__device__ __forceinline__ cxd electric_pair(const DevConst& dc, int pf, int l, const T* W, int lane, double gval,
                                             ElectricShared<H>& sh) {
    typename Wide<T>::Z w[2 * H];
    int a0, b0;
    link_ends(dc.g, l, a0, b0);
    electric_load<T, H>(dc, pf, l, a0, b0, W, lane, gval, sh, w);
    __syncwarp();
    electric_rows<T, H>(lane, w, sh);
    __syncwarp();
    electric_products<T, H>(dc, l, a0, lane, sh);
    __syncwarp();
    const cxd v = electric_value<T, H, FIELD>(dc.g, lane, sh);
    __syncwarp();
    return v;
}

// N_nm(G) / N(G) of chain c into out[c][n][m] for every ordered pair.
__host__ __device__ inline void pair_norm_item(const DevConst& dc, int c, const cxd* ell, cxd* out) {
    const int K = dc.K;
    const cxd* el = ell + (size_t)c * dc.P;
    double amax, iden;
    pair_scale(dc, el, amax, iden);
    cxd* o = out + (size_t)c * K * K;
    for (int p = 0; p < dc.P; ++p) {
        const cxd Np = pair_norm(dc, el, p, amax, iden);
        int n, m;
        pair_nm(K, p, n, m);
        o[n * K + m] = Np;
        if (n != m) o[m * K + n] = conjg(Np);
    }
}

// ---- fermionic (the derivation is in k_fermion.cu) ---------------------------

GGF_HD cxd times_minus_i(cxd v) { return {v.y, -v.x}; }

// Per-pair expectation -i (A + X)[alpha][beta] of entry (alpha, beta) of item
// (s, t), with c_a c_a = 1 where both Majoranas coincide (self-links).
GGF_HD cxd pair_bilinear(const DevConst& dc, int s, int t, int a, int b, cxd x) {
    if (s == t) {
        if (a == b) return cxd{1.0, 0.0};
        x.x += dc.Ap[(size_t)s * 4 + a * 2 + b];
    }
    return times_minus_i(x);
}

// What lane `lane` of the BW of item it of chain c keeps: entry (a, b) of the
// block of sites (s, t), each held by BW / 4 lanes of which the first writes, and where it goes in the combined and in
// the per-pair outputs (items 0 .. V - 1 are sites, of which only the entry
// (0, 1) is kept, then the links).
struct FermionLane {
    bool is_site, entry;
    int s, t, a, b;
    size_t out, pair;
};
template <int BW>
GGF_HD FermionLane fermion_lane(const Geometry& g, int K, int c, int it, int lane) {
    FermionLane f;
    const int e = lane / (BW / 4);
    f.is_site = it < g.V;
    f.s = f.t = it;
    if (!f.is_site) {
        int a0, b0;
        link_ends(g, it - g.V, a0, b0);
        f.s = a0 / g.B;
        f.t = b0 / g.B;
    }
    f.a = e >> 1;
    f.b = e & 1;
    f.entry = lane % (BW / 4) == 0 && (!f.is_site || e == 1);
    f.out = f.is_site ? (size_t)c * g.V + f.s : ((size_t)c * g.n_links + (it - g.V)) * 4 + e;
    f.pair = f.is_site ? f.out * K * K : (((size_t)c * g.n_links + (it - g.V)) * 4 + (f.a * 2 + f.b)) * K * K;
    return f;
}

// Pair p's block entry x (norm Np, weight E) into the lane's sum, and its two
// orders into the per-pair output q [K][K] (or null): of a complex pair
// (n, m) with weight E / 2 (w_p = 2 lambda_n^* lambda_m), (m, n) with conj(E) / 2
// and the conjugate product; A is added after the loop.
GGF_HD void fermion_term(const DevConst& dc, const FermionLane& f, int p, cxd Np, cxd E, cxd x, cxd& acc, cxd* q) {
    const cxd h = 0.5 * E;
    acc += h * x + conjg(h) * conjg(x);
    if (q) {
        int n, m;
        pair_nm(dc.K, p, n, m);
        q[n * dc.K + m] = Np * pair_bilinear(dc, f.s, f.t, f.a, f.b, x);
        q[m * dc.K + n] = conjg(Np) * pair_bilinear(dc, f.s, f.t, f.a, f.b, conjg(x));
    }
}
GGF_HD void fermion_term(const DevConst& dc, const FermionLane& f, int p, cxd Np, cxd E, double x, cxd& acc, cxd* q) {
    axpy(acc, x, E);
    if (q) q[p * dc.K + p] = Np * pair_bilinear(dc, f.s, f.t, f.a, f.b, cxd{x, 0.0});
}

// X[alpha][beta] = B_s W[s, t] B_t^T: row `lane` of the block's part of the sum.
template <class T, int BW>
GGF_HD void coupled_row(const DevConst& dc, const T* W, int s, int t, int lane, typename Wide<T>::Z (&X)[4]) {
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
}

// Entry (0, 1) of X on a site's own block: row `lane`'s part of the sum.
template <class T, int BW>
GGF_HD typename Wide<T>::Z coupled_row01(const DevConst& dc, const T* W, int s, int lane) {
    typedef typename Wide<T>::Z Z;
    const double* Bs = dc.Bp + (size_t)s * 2 * BW;
    Z w[BW], u1 = Sc<Z>::zero();
    load_run<BW>(W + (size_t)(s * BW + lane) * dc.g.N + (size_t)s * BW, w);
#pragma unroll
    for (int j = 0; j < BW; ++j) axpy(u1, Bs[BW + j], w[j]);
    return Bs[lane] * u1;
}

// Sums over the group's lanes: every round halves the values a lane carries as
// long as it has several, so that four values take 4 or 5 additions instead of
// 12 or 16 (the additions are those of a butterfly over all lanes).
template <class Z>
__device__ __forceinline__ Z fold_(Z low, Z high, int lane, int o) {
    const bool up = lane & o;
    return (up ? high : low) + shfl_xor_(up ? low : high, o);
}
__device__ __forceinline__ double from_lane_(double v, int src, int width) { return __shfl_sync(0xffffffffu, v, src, width); }
__device__ __forceinline__ cxd from_lane_(cxd v, int src, int width) {
    return {__shfl_sync(0xffffffffu, v.x, src, width), __shfl_sync(0xffffffffu, v.y, src, width)};
}

// The block product's entry lane / (BW / 4).
template <class T, int BW>
__device__ __forceinline__ typename Wide<T>::Z coupled_entry(const DevConst& dc, const T* W, int s, int t, int lane) {
    typedef typename Wide<T>::Z Z;
    Z X[4];
    coupled_row<T, BW>(dc, W, s, t, lane, X);
    const Z y0 = fold_(X[0], X[2], lane, BW / 2), y1 = fold_(X[1], X[3], lane, BW / 2);
    Z x = fold_(y0, y1, lane, BW / 4);
#pragma unroll
    for (int o = BW / 8; o > 0; o >>= 1) x = x + shfl_xor_(x, o);
    return x;
}

// What the four-point function of link (s, t) needs of a pair's inverse, in
// every lane of the group: X of (s, t), and its entries (0, 1) of (s, s) and (t, t).
template <class T, int BW>
__device__ __forceinline__ void four_point_blocks(const DevConst& dc, const T* W, int s, int t, int lane,
                                                  typename Wide<T>::Z& g01, typename Wide<T>::Z& g23,
                                                  typename Wide<T>::Z (&x)[4]) {
    typedef typename Wide<T>::Z Z;
    Z own = fold_(coupled_row01<T, BW>(dc, W, s, lane), coupled_row01<T, BW>(dc, W, t, lane), lane, BW / 2);
#pragma unroll
    for (int o = BW / 4; o > 0; o >>= 1) own = own + shfl_xor_(own, o);
    const Z e = coupled_entry<T, BW>(dc, W, s, t, lane);
    g01 = from_lane_(own, 0, BW);
    g23 = from_lane_(own, BW / 2, BW);
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = from_lane_(e, k * (BW / 4), BW);
}

// Pair p's part of <c_2s c_2s+1 c_2t c_2t+1> on link (s, t), from the blocks
// (s, s), (t, t) (entries 0 1) and (s, t): per pair, Wick's theorem gives
// Pf(-i G4) = -Pf(G4) with G4 the physical covariance A + B W B^T on those four
// Majoranas ((t, s) = -(s, t)^T), and the pairs combine with lambda_n^* lambda_m
// N_nm / N(G) as for the bilinears.  Lane 0: (n, m) with E / 2, lane 1: (m, n)
// with conj(E) / 2 and the conjugate blocks; a diagonal pair once with E.  A
// self-link (s = t) gives c_2s c_2s+1 c_2s c_2s+1 = -1.
GGF_HD void four_point_term(const DevConst& dc, int p, int lane, int s, int t, cxd g01, cxd g23, const cxd (&x)[4],
                            cxd Np, cxd E, cxd& acc, cxd* q) {
    if (lane > 1) return;
    const bool ord = lane == 1;
    const double As = dc.Ap[(size_t)s * 4 + 1], At = dc.Ap[(size_t)t * 4 + 1];
    auto cj = [&](cxd v) { return ord ? conjg(v) : v; };
    const cxd pf = (cj(g01) + cxd{As, 0.0}) * (cj(g23) + cxd{At, 0.0}) - cj(x[0]) * cj(x[3]) + cj(x[1]) * cj(x[2]);
    const cxd v = s == t ? cxd{1.0, 0.0} : pf;
    acc -= (0.5 * cj(E)) * v;
    if (q) {
        int n, m;
        pair_nm(dc.K, p, n, m);
        q[ord ? m * dc.K + n : n * dc.K + m] = -1.0 * (cj(Np) * v);
    }
}
GGF_HD void four_point_term(const DevConst& dc, int p, int lane, int s, int t, double g01, double g23,
                            const double (&x)[4], cxd Np, cxd E, cxd& acc, cxd* q) {
    if (lane > 0) return;
    const double As = dc.Ap[(size_t)s * 4 + 1], At = dc.Ap[(size_t)t * 4 + 1];
    const double pf = (g01 + As) * (g23 + At) - x[0] * x[3] + x[1] * x[2];
    const double v = s == t ? 1.0 : pf;
    axpy(acc, -v, E);
    if (q) q[p * dc.K + p] = -1.0 * (v * Np);
}

// ---- gauge-invariant link terms ------------------------------------------------
// A physical bilinear across link l = (s -> t) is gauge invariant together with
// the link operator u_l (Z2: g_l; U(1): e^{i theta_l}, diagonal in G) when it
// carries the charge u_l removes: T_l = u_l F_s F_t with F_s = psi_s (q_s > 0)
// or psi_s^dag (q_s < 0) and F_t = psi_t^dag (q_t > 0) or psi_t (q_t < 0); for
// staggered charges that is the pair term, and T_l + T_l^dag the link's hopping
// term.  With psi = (c_0 + i c_1) / 2 and the link block X[alpha][beta] =
// <c_{2s+alpha} c_{2t+beta}> (entries `stride` apart),
//   T_l = u_l (1/4) (X00 + i e_t X01 + i e_s X10 - e_s e_t X11),
// e = +1 for psi, -1 for psi^dag.
GGF_HD cxd link_term(const cxd* X, size_t stride, int e_s, int e_t, cxd u) {
    const cxd v = X[0] + cxd{0.0, (double)e_t} * X[stride] + cxd{0.0, (double)e_s} * X[2 * stride] +
                  (-(double)(e_s * e_t)) * X[3 * stride];
    return u * (0.25 * v);
}

// Chain c, link l: T_l from the combined link block blk [n][n_links][2][2]
// into out[c][l], and from the per-pair blocks pair_blk
// [n][n_links][2][2][K][K] into pair_out[c][l][n][m] (either pair of pointers
// may be null); q [V] the sites' physical charges.
GGF_HD void link_term_item(const DevConst& dc, int c, int l, const void* links, const int* q, const cxd* blk,
                           const cxd* pair_blk, cxd* out, cxd* pair_out) {
    const Geometry& g = dc.g;
    int a0, b0;
    link_ends(g, l, a0, b0);
    const int s = a0 / g.B, t = b0 / g.B;
    const int e_s = q[s] > 0 ? 1 : -1, e_t = q[t] > 0 ? -1 : 1;
    const size_t cl = (size_t)c * g.n_links + l;
    cxd u;
    if (g.group == GGF_Z2) {
        u = cxd{(double)((const int8_t*)links)[cl], 0.0};
    } else {
        const double th = ((const double*)links)[cl];
        u = cxd{cos(th), sin(th)};
    }
    if (blk && out) out[cl] = link_term(blk + cl * 4, 1, e_s, e_t, u);
    if (pair_blk && pair_out) {
        const int KK = dc.K * dc.K;
        for (int nm = 0; nm < KK; ++nm)
            pair_out[cl * KK + nm] = link_term(pair_blk + cl * 4 * KK + nm, (size_t)KK, e_s, e_t, u);
    }
}

// ---- score of the site blocks ------------------------------------------------
// d log N(G) / d D_s[i][j] of chain c and site s (entries treated as
// independent).  For pure site states N_nm(G) = const Pf(D + O Gamma_X O^T) and
// d log Pf(M) = (1/2) tr(M^{-1} dM), so the score is Re sum_p w_p (N_p / N(G))
// (1/2) W_p[s, s]^T (the (m, n) order of a pair n < m is the conjugate term,
// hence the real part): entry (i, j) from W_p[s B + j][s B + i].
template <class RW, class CW, int B>
GGF_HD double score_entry(const DevConst& dc, int c, int s, int i, int j, const RW* Wr, const CW* Wc,
                          const cxd* Es) {
    const Geometry& g = dc.g;
    const int K = dc.K;
    const size_t NN = (size_t)g.N * g.N, off = (size_t)(s * B + j) * g.N + (size_t)s * B + i;
    double acc = 0.0;
    for (int p = 0; p < dc.P; ++p) {
        const cxd E = Es[p];
        if (p < K) {
            acc = fma(0.5 * E.x, widen(Wr[((size_t)c * K + p) * NN + off]), acc);
        } else {
            const cxd w = widen(Wc[((size_t)c * dc.Kc + (p - K)) * NN + off]);
            acc = fma(0.5 * E.x, w.x, acc);
            acc = fma(-0.5 * E.y, w.y, acc);
        }
    }
    return acc;
}

// ---- score of the link blocks ------------------------------------------------
// Pair p, link l of chain c: out[c][p][l] (R x R complex, R = r) =
// (w_p N_p / N(G)) (1/2) (O_l^T W_p[l, l] O_l)^T with W_p[l, l] the block of the
// pair's inverse on the link's Majoranas and O_l the link's twist, so that
// d log N(G) = Re sum_p sum_l tr(U_p[l]^T dGamma_X^p[l]) + the pair constants'
// terms (none for K = 1, where this is the gradient for the bond blocks).  One
// warp per (chain, pair, link), in phases.

// Phase 1: the source end's rotation, rows O[x][a] (H x H).
template <int H>
GGF_HD void link_score_twist(const DevConst& dc, const void* links, int c, int l, int lane, double* O) {
    const Geometry& g = dc.g;
    if (g.group == GGF_SU2) {
        if (lane == 0) doublet_rotation(link_quat(g, links, c, l), O);
    } else if (lane < H) {
        double gval, theta, cs = 1.0, sn = 0.0;
        link_value<double>(dc, links, c, l, gval, theta);
        if (g.group == GGF_U1) sincos(g.q[lane >> 1] * theta, &sn, &cs);
        int i0, i1;
        double c0, c1;
        twist_row(g, lane, gval, cs, sn, i0, c0, i1, c1);
        for (int a = 0; a < H; ++a) O[lane * H + a] = 0.0;
        O[lane * H + i0] = c0;
        if (i1 != i0) O[lane * H + i1] = c1;
    }
}

// Phase 2: the block of W.
template <class T, int R>
GGF_HD void link_score_load(const DevConst& dc, const T* W, int l, int lane, cxd* w) {
    int a0, b0;
    link_ends(dc.g, l, a0, b0);
    for (int e = lane; e < R * R; e += 32)
        w[e] = as_cx(widen(W[(size_t)link_majorana(dc.g, a0, b0, e / R) * dc.g.N + link_majorana(dc.g, a0, b0, e % R)]));
}

// Phase 3: W O (the twist mixes the source-end columns only), kept by the lanes.
template <int R> struct LinkScoreRow { cxd t[(R * (R / 2) + 31) / 32]; };
template <int R>
GGF_HD void link_score_mix(const double* O, const cxd* w, int lane, LinkScoreRow<R>& m) {
    constexpr int H = R / 2;
    int k = 0;
    for (int e = lane; e < R * H; e += 32, ++k) {
        m.t[k] = cxd{0.0, 0.0};
        for (int b = 0; b < H; ++b) axpy(m.t[k], O[b * H + e % H], w[(e / H) * R + b]);
    }
}

// Phase 4: back into the block.
template <int R>
GGF_HD void link_score_put(int lane, const LinkScoreRow<R>& m, cxd* w) {
    constexpr int H = R / 2;
    int k = 0;
    for (int e = lane; e < R * H; e += 32, ++k) w[(e / H) * R + e % H] = m.t[k];
}

// Phase 5: out[x][y] = f (O^T W O)[y][x].
template <int R>
GGF_HD void link_score_out(const double* O, const cxd* w, cxd f, int lane, cxd* o) {
    constexpr int H = R / 2;
    for (int e = lane; e < R * R; e += 32) {
        const int x = e / R, y = e % R;
        cxd v = w[y * R + x];
        if (y < H) {
            v = cxd{0.0, 0.0};
            for (int a = 0; a < H; ++a) axpy(v, O[a * H + y], w[a * R + x]);
        }
        o[e] = f * v;
    }
}

}  // namespace
