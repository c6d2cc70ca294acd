// Metropolis sweep kernels of libggf (Sec. 5.1 sampling of p(G) = N(G)/N).
//
// Per link step, for every chain in lockstep:
//  ratio_kernel   one cluster per chain.  Draws the Philox numbers, forms the
//                 change Delta of the twisted link block for every pair
//                 (n, m), gathers W_SS from the cached inverse W = M^{-1},
//                 evaluates the Pfaffian ratio
//                    Pf(M') / Pf(M) = Pf([[Delta, -1], [1, W_SS]])
//                 (r/2 = 2 n_v even, so no extra sign) warp-parallel in FP64,
//                 combines the pairs into N(G')/N(G), decides, and on accept
//                 writes Z = (1 + Delta W_SS)^{-1} Delta, the rows Y = W[S, :]
//                 and the columns C = W[:, S].
//  update_kernel  rank-r Sherman-Morrison-Woodbury update of every pair's W
//                 of the accepted chains:  W <- W - C Z Y.
//                 The columns are gathered explicitly: replacing C by -Y^T
//                 (exact for an antisymmetric W) lets the rounding error's
//                 symmetric part grow geometrically from update to update.
//  observe_kernel per sweep: plaquette mean, log N(G), acceptance rate.
#include <cooperative_groups.h>
#include "ggf_ctx.h"
#include "ggf_geom.cuh"

#include "ggf_sweep.cuh"

namespace cg = cooperative_groups;

namespace {

struct SweepArgs {
    DevConst dc;
    int n_chains;
    const unsigned long long* d_sweep;   // sweep index (device, so captured sweeps replay)
    int link;
    uint64_t seed;
    uint64_t coff;         // Philox key word 1 = coff + chain
    double width;
    void* links;
    const void* Wr;
    const void* Wc;
    cxd* ell;
    cxd* zbuf;
    void* ybuf_r;
    void* ybuf_c;
    int* accept;
    int* since_refresh;
    int* sweep_acc;
    unsigned long long* counters;
    // delayed updates
    const void* Pr;   // real-family panels  [n][K][2][N][KRM]
    const void* Pc;   // complex-family panels [n][Kc][2][2][N][KRM]
    int* pend;
    int kmax;   // > 1: delayed
    // block moves: per-chain link, forced new angle prop[c][32] entry k, dead flags
    const int* link_of_chain;
    const double* forced;
    int forced_k;
    int* dead;
    PairBins bins;
    unsigned char early[MAXCS];     // immediate mode: CTA b copies beside the Pfaffian (copy_early)
};

// 16-byte pieces of a run of reals
template <int n>
__device__ __forceinline__ void load_reals(const float* p, float* o) {
#pragma unroll
    for (int k = 0; k < n; k += 4) {
        const float4 v = *(const float4*)(p + k);
        o[k] = v.x; o[k + 1] = v.y; o[k + 2] = v.z; o[k + 3] = v.w;
    }
}
template <int n>
__device__ __forceinline__ void load_reals(const double* p, double* o) {
#pragma unroll
    for (int k = 0; k < n; k += 2) {
        const double2 v = *(const double2*)(p + k);
        o[k] = v.x; o[k + 1] = v.y;
    }
}
template <int n>
__device__ __forceinline__ void store_reals(float* p, const float* o) {
#pragma unroll
    for (int k = 0; k < n; k += 4) *(float4*)(p + k) = make_float4(o[k], o[k + 1], o[k + 2], o[k + 3]);
}
template <int n>
__device__ __forceinline__ void store_reals(double* p, const double* o) {
#pragma unroll
    for (int k = 0; k < n; k += 2) *(double2*)(p + k) = make_double2(o[k], o[k + 1]);
}
__device__ __forceinline__ double real_of(double v) { return v; }
__device__ __forceinline__ float real_of(float v) { return v; }
template <class Q> __device__ __forceinline__ Q real_of(cx<Q> v) { return v.x; }
__device__ __forceinline__ double imag_of(double) { return 0.0; }
__device__ __forceinline__ float imag_of(float) { return 0.f; }
template <class Q> __device__ __forceinline__ Q imag_of(cx<Q> v) { return v.y; }
template <class T, class Q> __device__ __forceinline__ T from_parts(Q x, Q y) {
    if constexpr (Sc<T>::CPLX) return T{x, y};
    else return x;
}

// n consecutive rank columns (n a multiple of the 16-byte piece, within one
// chunk of eight) of one panel row
template <class T, int n>
__device__ __forceinline__ void panel_load(const typename Sc<T>::R* p, size_t plane, T* o) {
    typename Sc<T>::R re[n], im[n];
    load_reals<n>(p, re);
    if constexpr (Sc<T>::CPLX) load_reals<n>(p + plane, im);
#pragma unroll
    for (int k = 0; k < n; ++k) o[k] = from_parts<T>(re[k], Sc<T>::CPLX ? im[k] : re[k]);
}
template <class T, int n>
__device__ __forceinline__ void panel_store(typename Sc<T>::R* p, size_t plane, const T* o) {
    typename Sc<T>::R re[n], im[n];
#pragma unroll
    for (int k = 0; k < n; ++k) { re[k] = real_of(o[k]); im[k] = imag_of(o[k]); }
    store_reals<n>(p, re);
    if constexpr (Sc<T>::CPLX) store_reals<n>(p + plane, im);
}

// Byte offsets of ratio_kernel's shared arrays.
struct RatioLayout {
    size_t rho, term, tw, pair, task, part, stage, total;
    size_t pair_bytes, task_bytes;
};
__host__ __device__ inline RatioLayout ratio_layout(int P, int r, int np, int KRM, size_t cw) {
    RatioLayout s;
    size_t o = 0;
    auto take = [&](size_t& at, size_t bytes) { at = o; o = (o + bytes + 15) & ~(size_t)15; };
    take(s.rho, (size_t)P * sizeof(cxd));
    take(s.term, (size_t)P * sizeof(cxd));
    take(s.tw, 36 * sizeof(double));
    s.pair_bytes = (size_t)3 * r * r * sizeof(cxd);            // Delta, W_SS, Z
    take(s.pair, np * s.pair_bytes);
    s.task_bytes = (size_t)(4 * r * r + r) * sizeof(cxd);      // bordered matrix or [A | B], a column
    take(s.task, (size_t)(2 * np < NWARP ? 2 * np : NWARP) * s.task_bytes);
    take(s.part, KRM ? (size_t)(NWARP * 32) * sizeof(cxd) : 0);
    take(s.stage, KRM ? (size_t)2 * r * (KRM + 1) * cw : 0);    // pending rows of U and V on S
    s.total = o;
    return s;
}

// W_SS of one pair (FP64, shared), less the pending updates where there are
// any: W_eff[S, S] = W[S, S] - U[S, :] V[:, S].  The pending rows on S are
// staged once, and the sums of an entry are split over the CTA's threads.
template <class T, int R>
__device__ __forceinline__ void load_wss(const Geometry& g, int a0, int b0, const T* W, typename Fp64Of<T>::Z* Ws) {
    for (int e = threadIdx.x; e < R * R; e += NWARP * 32)
        Ws[e] = wide(W[(size_t)link_majorana(g, a0, b0, e / R) * g.N + link_majorana(g, a0, b0, e % R)]);
}
template <class T, int R>
__device__ __forceinline__ void subtract_pending(const Geometry& g, int a0, int b0, const typename Sc<T>::R* U, size_t NK,
                                                 int NP, int kr, void* stage, void* part, typename Fp64Of<T>::Z* Ws) {
    typedef typename Fp64Of<T>::Z Z;
    constexpr int PARTS = NWARP * 32 / (R * R);
    const typename Sc<T>::R* Vt = U + PanelIO<T>::PLANES * NK;
    const int ld = kr + 1;
    T* Us = (T*)stage;
    T* Vs = Us + (size_t)R * ld;
    for (int e = threadIdx.x; e < R * kr; e += NWARP * 32) {
        const int x = e / kr, q = e - x * kr;
        const size_t at = pidx(link_majorana(g, a0, b0, x), q, NP);
        Us[x * ld + q] = PanelIO<T>::ld(U, NK, at);
        Vs[x * ld + q] = PanelIO<T>::ld(Vt, NK, at);
    }
    __syncthreads();
    Z* ps = (Z*)part;
    {
        const int en = threadIdx.x % (R * R), pt = threadIdx.x / (R * R);
        const T* u = Us + (en / R) * ld;
        const T* v = Vs + (en % R) * ld;
        Z acc = Sc<Z>::zero();
        for (int q = pt; q < kr; q += PARTS) fmac(acc, wide(u[q]), wide(v[q]));
        ps[threadIdx.x] = acc;
    }
    __syncthreads();
    if (threadIdx.x < R * R) {
        Z acc = ps[threadIdx.x];
        for (int k = 1; k < PARTS; ++k) acc += ps[k * R * R + threadIdx.x];
        Ws[threadIdx.x] -= acc;
    }
    __syncthreads();
}

// Rows Y = W[S, :] and columns C^T = W[:, S]^T of one pair into yb [2][R][N],
// by `cnt` threads from `first`.
template <class T, int R>
__device__ __forceinline__ void gather_rows_cols(int N, int a0, int b0, const T* W, T* yb, int first, int cnt) {
    constexpr int H = R / 2, E = 16 / sizeof(T);
    const int pieces = N / E;                       // N is a multiple of 8
    for (int e = first; e < R * pieces; e += cnt) {
        const int xi = e / pieces, k = e - xi * pieces;
        const int gi = xi < H ? a0 + xi : b0 + xi - H;
        ((float4*)(yb + (size_t)xi * N))[k] = ((const float4*)(W + (size_t)gi * N))[k];
    }
    for (int e = first; e < 2 * N; e += cnt) {
        const int end = e >= N, j = end ? e - N : e;
        const T* src = W + (size_t)j * N + (end ? b0 : a0);
#pragma unroll
        for (int k = 0; k < H; ++k) yb[(size_t)(R + end * H + k) * N + j] = src[k];
    }
}

// One proposal of every chain; a cluster per chain, its pairs dealt to the CTAs
// (deal_pairs).  The Pfaffian ratio and Z of a pair run side by side on two
// warps, the pair terms on the last one, and in immediate mode the warps in
// between already copy the rows and columns that an accepted update needs,
// where that is done before the Pfaffian is (copy_early).
// Bound: the latency of that chain of FP64 steps; one CTA that drew, formed
// Delta, W_SS, ratio, terms, Z and copies in turn took 134 us for 1024 chains of
// 8 x 8 Z2 and 185 us for a block-move link of 32 chains of 8 x 8 U(1), K = 2;
// 78 and 53 us so.
// SU2: SU(2) links (quaternion proposal and doublet twist); the Z2 and U(1)
// instantiations (SU2 = false) do not contain that code.
template <class RW, class CW, bool SU2, int R>
__global__ void __launch_bounds__(NWARP * 32, 2) ratio_kernel(SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smr[];
    typedef typename Sc<RW>::R QR;
    const Geometry& g = a.dc.g;
    const int P = a.dc.P, K = a.dc.K, Kc = P - K, N = g.N, KRM = a.kmax > 1 ? a.kmax * R : 0;
    const int CS = cg::this_cluster().num_blocks(), rank = cg::this_cluster().block_rank();
    const int c = blockIdx.x / CS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p0 = a.bins.first[rank], np = a.bins.first[rank + 1] - p0;
    const RatioLayout lay = ratio_layout(P, R, np, KRM, sizeof(CW));
    cxd* rho = (cxd*)(smr + lay.rho);
    cxd* term = (cxd*)(smr + lay.term);
    double* tw = (double*)(smr + lay.tw);
    auto slot = [&](int s, int k) { return (cxd*)(smr + lay.pair + s * lay.pair_bytes) + k * R * R; };
    __shared__ Proposal s_q;
    __shared__ int s_accept, s_okz[MAXP];

    const int l = a.link_of_chain ? a.link_of_chain[c] : a.link;
    const int dead = a.forced ? a.dead[c] : 0;
    const int kr = KRM ? a.pend[c] * R : 0;
    int a0, b0;
    link_ends(g, l, a0, b0);
    auto w_real = [&](int p) { return (const RW*)a.Wr + ((size_t)c * K + p) * N * N; };
    auto w_cplx = [&](int p) { return (const CW*)a.Wc + ((size_t)c * Kc + (p - K)) * N * N; };

    if (threadIdx.x == 0) {
        Proposal q{};
        if constexpr (SU2) {
            q.u_acc = draw_su2(g, a.links, c, l, *a.d_sweep, a.seed, a.width, tw, tw + 4, tw + 20, a.coff);
        } else {
            q = draw_proposal(g, a.links, c, l, *a.d_sweep, a.seed, a.width, a.coff);
            if (a.forced && g.group == GGF_U1) q.th_new = a.forced[(size_t)c * 32 + a.forced_k];   // block move
            if (g.group == GGF_U1)
                for (int t = 0; t < 2 * g.n_v; ++t) {
                    const int md = t % g.n_v, nw = t / g.n_v;
                    double sv, cv;
                    sincos(g.q[md] * (nw ? q.th_new : q.th_old), &sv, &cv);
                    tw[4 * nw + 2 * md] = cv;
                    tw[4 * nw + 2 * md + 1] = sv;
                }
        }
        s_q = q;
    }
    for (int s = 0; s < np; ++s) {
        const int p = a.bins.ord[p0 + s];
        if (p < K) load_wss<RW, R>(g, a0, b0, w_real(p), (double*)slot(s, 1));
        else load_wss<CW, R>(g, a0, b0, w_cplx(p), slot(s, 1));
    }
    __syncthreads();
    const Proposal q = s_q;
    const size_t NK = panel_plane(N, KRM ? KRM : R);
    const int NP = panel_rows(N);
    for (int s = 0; s < np; ++s) {
        const int p = a.bins.ord[p0 + s];
        if (kr > 0) {
            if (p < K)
                subtract_pending<RW, R>(g, a0, b0, (const QR*)a.Pr + ((size_t)c * K + p) * 2 * NK, NK, NP, kr,
                                        smr + lay.stage, smr + lay.part, (double*)slot(s, 1));
            else
                subtract_pending<CW, R>(g, a0, b0, (const QR*)a.Pc + ((size_t)c * Kc + (p - K)) * 4 * NK, NK, NP, kr,
                                        smr + lay.stage, smr + lay.part, slot(s, 1));
        }
        for (int e = threadIdx.x; e < R * R; e += NWARP * 32) {
            if (p < K) ((double*)slot(s, 0))[e] = delta_elem<double>(a.dc, p, l, e / R, e % R, q, tw, SU2);
            else slot(s, 0)[e] = delta_elem<cxd>(a.dc, p - K, l, e / R, e % R, q, tw, SU2);
        }
    }
    // every CTA of the cluster is running before the first remote write
    if (CS > 1) cg::this_cluster().sync();
    else __syncthreads();

    const int spare0 = min(2 * np, NWARP - 1), spare = NWARP - 1 - spare0;
    if (warp == NWARP - 1) {
        double amax = -INFINITY;
        for (int p = lane; p < P; p += 32) amax = fmax(amax, a.dc.logc[p].x + a.ell[(size_t)c * P + p].x);
        for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        for (int p = lane; p < P; p += 32) {
            cxd e = a.dc.logc[p] + a.ell[(size_t)c * P + p];
            if (p < K) e.y = 0.0;
            e.x -= amax;
            term[p] = a.dc.w[p] * cexp_(e);
        }
    }
    for (int t = warp; t < 2 * np; t += NWARP) {
        const int s = t >> 1, p = a.bins.ord[p0 + s];
        void* scr = smr + lay.task + (size_t)warp * lay.task_bytes;
        if (t & 1) {
            const bool ok = p < K ? pair_z<sizeof(RW) == 4>((const double*)slot(s, 0), (const double*)slot(s, 1), (double*)scr,
                                           (double*)scr + 4 * R * R, R, slot(s, 2))
                                  : pair_z<sizeof(RW) == 4>(slot(s, 0), slot(s, 1), (cxd*)scr, (cxd*)scr + 4 * R * R, R, slot(s, 2));
            if (lane == 0) s_okz[s] = ok;
        } else {
            const cxd pf = p < K ? cxd{bordered_ratio((const double*)slot(s, 0), (const double*)slot(s, 1), (double*)scr, R), 0.0}
                                 : bordered_ratio(slot(s, 0), slot(s, 1), (cxd*)scr, R);
            if (lane < CS) {
                cxd* dst = rho + p;
                if (CS > 1) dst = cg::this_cluster().map_shared_rank(dst, lane);
                *dst = pf;
            }
            __syncwarp();
        }
    }
    auto copy_rows = [&](int first, int cnt) {
        for (int s = 0; s < np; ++s) {
            const int p = a.bins.ord[p0 + s];
            if (p < K) gather_rows_cols<RW, R>(N, a0, b0, w_real(p), (RW*)a.ybuf_r + ((size_t)c * K + p) * 2 * R * N, first, cnt);
            else gather_rows_cols<CW, R>(N, a0, b0, w_cplx(p), (CW*)a.ybuf_c + ((size_t)c * Kc + (p - K)) * 2 * R * N, first, cnt);
        }
    };
    if (a.early[rank] && warp >= spare0 && warp < NWARP - 1)
        copy_rows((warp - spare0) * 32 + lane, spare * 32);
    if (CS > 1) cg::this_cluster().sync();
    else __syncthreads();

    if (warp == 0) {
        int acc;
        if (a.forced) {
            // block move: every link of the block is taken tentatively; the move is
            // decided once the whole block's ratio is known
            bool ok = dead == 0;
            for (int p = lane; p < P; p += 32) ok = ok && is_fin(rho[p]) && !is_zero(rho[p]);
            acc = __all_sync(0xffffffffu, ok) ? 1 : 0;
        } else {
            double so = 0.0, sn = 0.0;
            for (int p = lane; p < P; p += 32) {
                so += term[p].x;
                sn += (term[p] * rho[p]).x;
            }
            for (int o = 16; o > 0; o >>= 1) {
                so += __shfl_xor_sync(0xffffffffu, so, o);
                sn += __shfl_xor_sync(0xffffffffu, sn, o);
            }
            acc = (sn > 0.0 && so > 0.0 && q.u_acc < sn / so) ? 1 : 0;
        }
        if (lane == 0) s_accept = acc;
        if (rank == 0 && lane == 0) {
            a.accept[c] = acc;
            if (a.forced) {
                if (!acc) a.dead[c] = 1;
            } else {
                atomicAdd(&a.counters[0], 1ULL);
            }
            if (acc) {
                if (a.kmax > 1) a.pend[c] += 1;
                if (!a.forced) {
                    atomicAdd(&a.counters[1], 1ULL);
                    a.since_refresh[c] += 1;
                    a.sweep_acc[c] += 1;
                }
                if constexpr (SU2) {
                    double* dst = (double*)a.links + ((size_t)c * g.n_links + l) * 4;
                    for (int k = 0; k < 4; ++k) dst[k] = tw[k];
                } else {
                    if (g.group == GGF_Z2) ((int8_t*)a.links)[(size_t)c * g.n_links + l] = (int8_t)q.g_new;
                    else ((double*)a.links)[(size_t)c * g.n_links + l] = q.th_new;
                }
            }
        }
    }
    __syncthreads();
    if (!s_accept) return;
    if (rank == 0 && warp == NWARP - 1)
        for (int p = lane; p < P; p += 32) ell_add(a.ell[(size_t)c * P + p], rho[p], p < K);
    for (int s = 0; s < np; ++s) {
        const int p = a.bins.ord[p0 + s];
        for (int e = threadIdx.x; e < R * R; e += NWARP * 32) a.zbuf[((size_t)c * P + p) * R * R + e] = slot(s, 2)[e];
        if (!s_okz[s] && a.forced && threadIdx.x == 0) a.dead[c] = 1;
    }
    // (delayed mode: gather_kernel forms the rows and columns)
    if (a.kmax <= 1 && !a.early[rank]) copy_rows(threadIdx.x, NWARP * 32);
}

// W <- W - C Z Y of the accepted chains.  Bound: the traffic of W, read and
// written once; each thread takes 16 bytes of a row and four rows at a time, so
// that four independent loads are in flight (one element of one row at a time
// moved 3.6 TB/s: 1024 chains of 8 x 8 Z2, of which 92 % accept, took 542 us
// per link, 294 us so, 6.7 TB/s).
template <class T, int R>
__global__ void __launch_bounds__(256) update_kernel(int N, int P, int fam_pairs, int pair_off, T* W,
                                                     const T* ybuf, const cxd* zbuf, const int* accept, int TI) {
    const int c = blockIdx.z;
    if (!accept[c]) return;
    const int p = blockIdx.y;
    extern __shared__ unsigned char smraw[];
    T* Zs = (T*)smraw;        // [R][R]
    T* Pr = Zs + R * R;       // [TI][R]
    T* Wp = W + ((size_t)c * fam_pairs + p) * N * N;
    const T* Y = ybuf + ((size_t)c * fam_pairs + p) * 2 * R * N;   // rows W[S, :]
    const T* Ct = Y + (size_t)R * N;                                 // columns W[:, S]^T
    const cxd* Z = zbuf + ((size_t)c * P + pair_off + p) * R * R;
    for (int e = threadIdx.x; e < R * R; e += blockDim.x) Zs[e] = Sc<T>::from(Z[e]);
    __syncthreads();
    const int i0 = blockIdx.x * TI;
    const int ti = min(TI, N - i0);
    for (int e = threadIdx.x; e < ti * R; e += blockDim.x) {
        int i = e / R, b = e % R;
        T acc = Sc<T>::zero();
#pragma unroll
        for (int q = 0; q < R; ++q) acc += Ct[(size_t)q * N + i0 + i] * Zs[q * R + b];
        Pr[i * R + b] = acc;
    }
    __syncthreads();
    constexpr int E = 16 / sizeof(T);       // elements per piece; N is a multiple of 8
    const int pieces = N / E, width = min(pieces, 256), rows = 256 / width;
    const int t = threadIdx.x % width, r0 = threadIdx.x / width;
    if (r0 >= rows) return;
    union Piece { float4 v; T e[E]; };
    for (int k = t; k < pieces; k += width) {
        T y[R][E];
#pragma unroll
        for (int b = 0; b < R; ++b) {
            Piece u;
            u.v = ((const float4*)(Y + (size_t)b * N))[k];
#pragma unroll
            for (int x = 0; x < E; ++x) y[b][x] = u.e[x];
        }
        for (int i = r0; i < ti; i += 4 * rows) {
            Piece w[4];
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (i + m * rows < ti) w[m].v = ((const float4*)(Wp + (size_t)(i0 + i + m * rows) * N))[k];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int ii = i + m * rows;
                if (ii >= ti) break;
#pragma unroll
                for (int x = 0; x < E; ++x) {
                    T acc = w[m].e[x];
#pragma unroll
                    for (int b = 0; b < R; ++b) acc -= Pr[ii * R + b] * y[b][x];
                    w[m].e[x] = acc;
                }
                ((float4*)(Wp + (size_t)(i0 + ii) * N))[k] = w[m].v;
            }
        }
    }
}

// Products of the block-move gather.  FP32 complex ones with their roundings
// written out (which of the two terms of the imaginary part is rounded first
// shows in the last bit of the panels, and through a block move's low-weight
// configurations far above it): im = fma(ax, by, ay bx) for MF = false,
// fma(ay, bx, ax by) for MF = true; re = fma(ax, bx, -(ay by)).
template <bool MF, class T> __device__ __forceinline__ T gather_mul(T a, T b) {
    if constexpr (sizeof(T) == sizeof(cxf) && Sc<T>::CPLX) {
        T r;
        r.x = __fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y));
        r.y = MF ? __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)) : __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x));
        return r;
    } else {
        return a * b;
    }
}
template <bool MF, class T> __device__ __forceinline__ void gather_sub(T& r, T a, T b) {
    if constexpr (sizeof(T) == sizeof(cxf) && Sc<T>::CPLX) {
        const T t = gather_mul<MF>(a, b);
        r = {__fsub_rn(r.x, t.x), __fsub_rn(r.y, t.y)};
    } else {
        acc_sub(r, a, b);
    }
}
template <bool MF, class T> __device__ __forceinline__ void gather_add(T& r, T a, T b) {
    if constexpr (sizeof(T) == sizeof(cxf) && Sc<T>::CPLX) {
        const T t = gather_mul<MF>(a, b);
        r = {__fadd_rn(r.x, t.x), __fadd_rn(r.y, t.y)};
    } else {
        acc_add(r, a, b);
    }
}

// Block moves, accepted chains: rows Y = W_eff[S, :] and columns
// C = W_eff[:, S] of the effective inverse W_eff = W - U V, then the new
// panel entries U[:, slot] = C Z and V[slot, :] = Y (stored as V^T rows).
// Grid (ceil(N / 128), pairs, chains), 128 threads, one index each: its panel
// rows are read straight from the chunk-major panels (eight rank columns of
// neighbouring rows are one run), the rows on S from shared memory.
// Bound: panel reads from L2 and FP32 arithmetic at high rank; with the panel
// rows staged element by element, and a launch per family, a block-move link of
// 32 chains of 8 x 8 U(1), K = 2 took 150 us, 59 so.
template <class T, int R>
__device__ __forceinline__ void gather_pair(const Geometry& g, const int* S, const T* Wp, typename Sc<T>::R* U,
                                            const cxd* Z, int kr, int KRM, unsigned char* smraw) {
    typedef typename Sc<T>::R RR;
    const int N = g.N, NP = panel_rows(N);
    const size_t NK = panel_plane(N, KRM);
    T* UtS = (T*)smraw;            // [kr][R]  U[S_a, q]
    T* VS = UtS + (size_t)KRM * R; // [kr][R]  V[q, S_a]
    T* Zs = VS + (size_t)KRM * R;  // [R][R]
    RR* Vt = U + PanelIO<T>::PLANES * NK;
    for (int e = threadIdx.x; e < kr * R; e += blockDim.x) {
        const int a = e / kr, q = e - a * kr;
        UtS[q * R + a] = PanelIO<T>::ld(U, NK, pidx(S[a], q, NP));
        VS[q * R + a] = PanelIO<T>::ld(Vt, NK, pidx(S[a], q, NP));
    }
    for (int e = threadIdx.x; e < R * R; e += blockDim.x) Zs[e] = Sc<T>::from(Z[e]);
    __syncthreads();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    T yv[R], cv[R];
#pragma unroll
    for (int a = 0; a < R; ++a) {
        yv[a] = Wp[(size_t)S[a] * N + j];
        cv[a] = Wp[(size_t)j * N + S[a]];
    }
    // R rank columns per step (kr is a multiple of R, and R of them stay within a
    // chunk), the next step's loaded before this one's products
    T un[R], vn[R];
    if (kr > 0) {
        panel_load<T, R>(U + pidx(j, 0, NP), NK, un);
        panel_load<T, R>(Vt + pidx(j, 0, NP), NK, vn);
    }
    for (int q0 = 0; q0 < kr; q0 += R) {
        T uq[R], vq[R];
#pragma unroll
        for (int k = 0; k < R; ++k) { uq[k] = un[k]; vq[k] = vn[k]; }
        if (q0 + R < kr) {
            const size_t at = pidx(j, q0 + R, NP);
            panel_load<T, R>(U + at, NK, un);
            panel_load<T, R>(Vt + at, NK, vn);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) {
#pragma unroll
            for (int a = 0; a < R; ++a) {
                gather_sub<false>(yv[a], UtS[(q0 + k) * R + a], vq[k]);
                gather_sub<true>(cv[a], uq[k], VS[(q0 + k) * R + a]);
            }
        }
    }
    T u[R];
#pragma unroll
    for (int b = 0; b < R; ++b) {
        u[b] = Sc<T>::zero();
#pragma unroll
        for (int a = 0; a < R; ++a) gather_add<true>(u[b], cv[a], Zs[a * R + b]);
    }
    const size_t at = pidx(j, kr, NP);
    panel_store<T, R>(U + at, NK, u);
    panel_store<T, R>(Vt + at, NK, yv);
}

template <class RW, class CW, int R>
__global__ void __launch_bounds__(128) gather_kernel(Geometry g, int K, int Kc, int link_all, const int* link_of_chain,
                                                     const RW* Wr, const CW* Wc, typename Sc<RW>::R* Pr,
                                                     typename Sc<RW>::R* Pc, const cxd* zbuf, const int* accept,
                                                     const int* pend, int kmax) {
    const int c = blockIdx.z;
    if (!accept[c]) return;
    const int p = blockIdx.y, N = g.N, P = K + Kc;
    const int kr = (pend[c] - 1) * R, KRM = kmax * R;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int S[R];
    int a0, b0;
    link_ends(g, link_of_chain ? link_of_chain[c] : link_all, a0, b0);
    if (threadIdx.x < R) S[threadIdx.x] = link_majorana(g, a0, b0, threadIdx.x);
    __syncthreads();
    const size_t NK = panel_plane(N, KRM), NN = (size_t)N * N;
    const cxd* Z = zbuf + ((size_t)c * P + p) * R * R;
    if (p < K)
        gather_pair<RW, R>(g, S, Wr + ((size_t)c * K + p) * NN, Pr + ((size_t)c * K + p) * 2 * NK, Z, kr, KRM, smraw);
    else
        gather_pair<CW, R>(g, S, Wc + ((size_t)c * Kc + (p - K)) * NN, Pc + ((size_t)c * Kc + (p - K)) * 4 * NK, Z, kr, KRM,
                           smraw);
}

// W <- W - U V over the pending panels (rank pend[c] * R), SIMT tiled product
// (FP64 chains, and FP32 when the tensor-core flush is not used).
// Grid (tiles_i * tiles_j, family pairs, chains), 256 threads as 16 x 16, each
// four rows by four columns (16 apart, so that neighbouring threads touch
// neighbouring elements) of a 64 x 64 tile of W.  Bound: the FP64 unit; with the
// complex product formed before it is added (six instructions instead of four
// fused ones) a rank-128 flush of 24 complex matrices of order 1024 took 35.3
// ms, 20.9 fused.
template <class T, int R>
__global__ void __launch_bounds__(256) flush_kernel(int N, int fam_pairs, T* W, const typename Sc<T>::R* Pan,
                                                    const int* pend, int kmax, int tiles) {
    typedef typename Sc<T>::R RR;
    const int c = blockIdx.z;
    const int kc = pend[c];
    if (kc == 0) return;
    const int kr = kc * R, KRM = kmax * R, NP = panel_rows(N);
    const size_t NK = panel_plane(N, KRM);
    const int p = blockIdx.y;
    const int ti = blockIdx.x / tiles, tj = blockIdx.x - ti * tiles;
    const int i0 = ti * 64, j0 = tj * 64;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    __shared__ T As[16][65];
    __shared__ T Bs[16][65];
    const size_t base = ((size_t)c * fam_pairs + p);
    T* Wp = W + base * N * N;
    const RR* U = Pan + base * 2 * PanelIO<T>::PLANES * NK;
    const RR* Vt = U + PanelIO<T>::PLANES * NK;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = Sc<T>::zero();
    for (int q0 = 0; q0 < kr; q0 += 16) {
        for (int e = threadIdx.x; e < 16 * 64; e += 256) {
            int k = e >> 4, qq = e & 15;      // consecutive threads walk the rank index
            int q = q0 + qq;
            As[qq][k] = (q < kr && i0 + k < N) ? PanelIO<T>::ld(U, NK, pidx(i0 + k, q, NP)) : Sc<T>::zero();
            Bs[qq][k] = (q < kr && j0 + k < N) ? PanelIO<T>::ld(Vt, NK, pidx(j0 + k, q, NP)) : Sc<T>::zero();
        }
        __syncthreads();
#pragma unroll
        for (int qq = 0; qq < 16; ++qq) {
            T av[4], bv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = As[qq][ty * 4 + a];
#pragma unroll
            for (int b = 0; b < 4; ++b) bv[b] = Bs[qq][tx + 16 * b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc_add(acc[a][b], av[a], bv[b]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        int i = i0 + ty * 4 + a;
        if (i >= N) continue;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int j = j0 + tx + 16 * b;
            if (j < N) Wp[(size_t)i * N + j] -= acc[a][b];
        }
    }
}

__global__ void reset_pend(int n, int* pend) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) pend[c] = 0;
}

__global__ void observe_kernel(DevConst dc, int n_chains, const void* links, const cxd* ell, const int* sweep_acc,
                               double* obs) {
    __shared__ double red[256];
    const Geometry& g = dc.g;
    int c = blockIdx.x;
    double acc = 0.0;
    for (int s = threadIdx.x; s < g.V; s += blockDim.x) {
        int x = s % g.L, y = s / g.L;
        int sx = y * g.L + (x + 1) % g.L, sy = ((y + 1) % g.L) * g.L + x;
        int l1 = 2 * s, l2 = 2 * sx + 1, l3 = 2 * sy, l4 = 2 * s + 1;
        if (g.group == GGF_Z2) {
            const int8_t* L8 = (const int8_t*)links + (size_t)c * g.n_links;
            acc += (double)(L8[l1] * L8[l2] * L8[l3] * L8[l4]);
        } else if (g.group == GGF_SU2) {
            acc += plaquette_su2(link_quat(g, links, c, l1), link_quat(g, links, c, l2), link_quat(g, links, c, l3),
                                 link_quat(g, links, c, l4));
        } else {
            const double* T = (const double*)links + (size_t)c * g.n_links;
            acc += cos(T[l1] + T[l2] - T[l3] - T[l4]);
        }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double amax = -INFINITY;
        for (int p = 0; p < dc.P; ++p) amax = fmax(amax, dc.logc[p].x + ell[(size_t)c * dc.P + p].x);
        double sv = 0.0;
        for (int p = 0; p < dc.P; ++p) {
            cxd e = dc.logc[p] + ell[(size_t)c * dc.P + p];
            if (p < dc.K) e.y = 0.0;
            e.x -= amax;
            sv += (dc.w[p] * cexp_(e)).x;
        }
        obs[(size_t)c * GGF_N_OBS + 0] = red[0] / g.V;
        obs[(size_t)c * GGF_N_OBS + 1] = sv > 0 ? amax + log(sv) : -INFINITY;
        obs[(size_t)c * GGF_N_OBS + 2] = (double)sweep_acc[c] / g.n_links;
    }
}

__global__ void mark_refresh(int n_chains, int R, const int* since, int* list) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_chains) return;
    if (since[c] >= R) {
        int k = atomicAdd(&list[0], 1);
        list[1 + k] = c;
    }
}

// Whether a CTA copies the rows and columns of its nr real and nc complex pairs
// before the decision, on `spare` warps beside the Pfaffian: only where the
// Pfaffian hides it, or a rejected proposal pays for a copy that nobody reads.
// The line is the loop trips of a spare thread (16-byte pieces of the rows,
// entries of the columns) against the order R of the blocks, in proportion to
// which the Pfaffian grows.  Microseconds per link, early and after
// the decision, accepted / rejected: 10 trips of R = 4 (8 x 8 Z2) 17 / 14 and
// 19 / 14, 26 of R = 8 (8 x 8 U(1), K = 1, FP32) 34 / 28 and 41 / 27, 32 (4 x 4
// U(1), K = 2, FP64) 48 / 36 and 52 / 33; but 38 of R = 4 (16 x 16 Z2) 41 / 27 and
// 37 / 15, 85 of R = 8 (8 x 8 U(1), K = 2, FP32) 83 / 64 and 70 / 40, 288
// (12 x 12, FP64) 202 / 185 and 118 / 33.  (Where the chains alone fill the chip,
// 1024 of 8 x 8 Z2, early is better from 75 % accepted on: 73 / 58 and 79 / 43.)
// rsz: bytes of a real element of W.
bool copy_early(int N, int R, int nr, int nc, int rsz) {
    const int spare = NWARP - 1 - std::min(2 * (nr + nc), NWARP - 1);
    const long long work = (long long)N * ((nr + 2 * nc) * R * rsz / 16 + 2 * (nr + nc));
    return spare > 0 && work <= 4LL * R * 32 * spare;
}

}  // namespace

ggf_status ggf_flush(ggf_ctx* ctx, cudaStream_t st);
ggf_status ggf_flush_tc(ggf_ctx* ctx, cudaStream_t st, int* launches);

ggf_status ggf_link_step_ex(ggf_ctx* ctx, int link, cudaStream_t st, const int* link_of_chain, const double* forced,
                            int forced_k, int* dead);

ggf_status ggf_link_step(ggf_ctx* ctx, int link, cudaStream_t st) {
    return ggf_link_step_ex(ctx, link, st, nullptr, nullptr, 0, nullptr);
}

// One proposal per chain.  Block moves pass a per-chain link, the proposed
// angles (forced, slot forced_k) and dead flags; the flush cadence then stays
// with the caller.
ggf_status ggf_link_step_ex(ggf_ctx* ctx, int link, cudaStream_t st, const int* link_of_chain, const double* forced,
                            int forced_k, int* dead) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    SweepArgs a;
    a.dc = ctx->dc();
    a.n_chains = ch.n;
    a.d_sweep = ch.d_sweep;
    a.link = link;
    a.seed = ch.opts.seed;
    a.coff = ch.opts.chain_offset;
    a.width = ch.opts.width;
    a.links = ch.links;
    a.Wr = ch.Wr;
    a.Wc = ch.Wc;
    a.ell = ch.ell;
    a.zbuf = (cxd*)ch.zbuf;
    const bool fp64 = ch.opts.precision == GGF_FP64;
    size_t rsz = fp64 ? sizeof(double) : sizeof(float);
    a.ybuf_r = ch.ybuf;
    a.ybuf_c = (unsigned char*)ch.ybuf + (size_t)ch.n * ctx->K * 2 * g.r * g.N * rsz;
    a.accept = ch.accept;
    a.since_refresh = ch.since_refresh;
    a.sweep_acc = ch.sweep_acc;
    a.counters = ch.counters;
    a.Pr = ch.Pr; a.Pc = ch.Pc;
    a.link_of_chain = link_of_chain;
    a.forced = forced;
    a.forced_k = forced_k;
    a.dead = dead;
    a.pend = ch.pend;
    a.kmax = ch.kmax;
    const int CS = deal_pairs(ctx->K, ctx->Kc, a.bins);
    size_t smem = 0;
    for (int b = 0; b < CS; ++b) {
        const int np = a.bins.first[b + 1] - a.bins.first[b];
        int nc = 0;
        for (int s = 0; s < np; ++s) nc += a.bins.ord[a.bins.first[b] + s] >= ctx->K;
        smem = std::max(smem, ratio_layout(ctx->P, g.r, np, ch.kmax > 1 ? ch.kmax * g.r : 0, 2 * rsz).total);
        a.early[b] = ch.kmax <= 1 && copy_early(g.N, g.r, np - nc, nc, (int)rsz);
    }
    const int ev0 = ctx->prof_mark(st);
    ctx->launches += 2 + (ctx->Kc ? 1 : 0);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ch.n * CS);
    cfg.blockDim = dim3(NWARP * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CS > 1 ? 1 : 0;
    if (g.group == GGF_SU2) {
        if (fp64) GGF_CK(cudaLaunchKernelEx(&cfg, ratio_kernel<double, cxd, true, 8>, a));
        else GGF_CK(cudaLaunchKernelEx(&cfg, ratio_kernel<float, cxf, true, 8>, a));
    } else if (g.r == 4) {
        if (fp64) GGF_CK(cudaLaunchKernelEx(&cfg, ratio_kernel<double, cxd, false, 4>, a));
        else GGF_CK(cudaLaunchKernelEx(&cfg, ratio_kernel<float, cxf, false, 4>, a));
    } else {
        if (fp64) GGF_CK(cudaLaunchKernelEx(&cfg, ratio_kernel<double, cxd, false, 8>, a));
        else GGF_CK(cudaLaunchKernelEx(&cfg, ratio_kernel<float, cxf, false, 8>, a));
    }
    const int ev1 = ctx->prof_mark(st);
    ctx->prof_pair(GGF_KT_RATIO, ev0, ev1);
    const int N = g.N;
    if (ch.kmax > 1) {
        dim3 gg((N + 127) / 128, ctx->P, ch.n);
#define GGF_GATH(RW, CW, R_)                                                                                         \
    gather_kernel<RW, CW, R_><<<gg, 128, (2 * (size_t)ch.kmax * R_ * R_ + R_ * R_) * sizeof(CW), st>>>(                \
        g, ctx->K, ctx->Kc, link, link_of_chain, (const RW*)ch.Wr, (const CW*)ch.Wc, (typename Sc<RW>::R*)ch.Pr,       \
        (typename Sc<RW>::R*)ch.Pc, a.zbuf, ch.accept, ch.pend, ch.kmax)
        if (g.r == 4) {
            if (fp64) GGF_GATH(double, cxd, 4); else GGF_GATH(float, cxf, 4);
        } else {
            if (fp64) GGF_GATH(double, cxd, 8); else GGF_GATH(float, cxf, 8);
        }
#undef GGF_GATH
        GGF_CK(cudaGetLastError());
        ctx->prof_pair(GGF_KT_UPDATE, ev1, ctx->prof_mark(st));
        if (forced) { ++ch.steps_since_flush; return GGF_OK; }
        if (++ch.steps_since_flush >= ch.kmax) GGF_TRY(ggf_flush(ctx, st));
        return GGF_OK;
    }
    // rows per CTA: 32 amortise its rank columns where they still fill the chip
    const int TI = (long long)ch.n * ctx->P * (N / 32) >= 8LL * ctx->n_sms ? 32 : 8;
    dim3 gr((N + TI - 1) / TI, ctx->K, ch.n);
    dim3 gc((N + TI - 1) / TI, ctx->Kc, ch.n);
#define GGF_UPD(T, R_, grid, fam, off, Wp, Yp)                                                         \
    update_kernel<T, R_><<<grid, 256, (R_ * R_ + TI * R_) * sizeof(T), st>>>(N, ctx->P, fam, off, (T*)(Wp), \
                                                                              (const T*)(Yp), a.zbuf, ch.accept, TI)
    if (g.r == 4) {
        if (fp64) {
            GGF_UPD(double, 4, gr, ctx->K, 0, ch.Wr, a.ybuf_r);
            if (ctx->Kc) GGF_UPD(cxd, 4, gc, ctx->Kc, ctx->K, ch.Wc, a.ybuf_c);
        } else {
            GGF_UPD(float, 4, gr, ctx->K, 0, ch.Wr, a.ybuf_r);
            if (ctx->Kc) GGF_UPD(cxf, 4, gc, ctx->Kc, ctx->K, ch.Wc, a.ybuf_c);
        }
    } else {
        if (fp64) {
            GGF_UPD(double, 8, gr, ctx->K, 0, ch.Wr, a.ybuf_r);
            if (ctx->Kc) GGF_UPD(cxd, 8, gc, ctx->Kc, ctx->K, ch.Wc, a.ybuf_c);
        } else {
            GGF_UPD(float, 8, gr, ctx->K, 0, ch.Wr, a.ybuf_r);
            if (ctx->Kc) GGF_UPD(cxf, 8, gc, ctx->Kc, ctx->K, ch.Wc, a.ybuf_c);
        }
    }
#undef GGF_UPD
    GGF_CK(cudaGetLastError());
    ctx->prof_pair(GGF_KT_UPDATE, ev1, ctx->prof_mark(st));
    return GGF_OK;
}

ggf_status ggf_flush(ggf_ctx* ctx, cudaStream_t st) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    if (ch.kmax <= 1 || ch.steps_since_flush == 0) return GGF_OK;
    const bool fp64 = ch.opts.precision == GGF_FP64;
    const int N = g.N, tiles = (N + 63) / 64;
    const int ev0 = ctx->prof_mark(st);
    dim3 gr(tiles * tiles, ctx->K, ch.n), gc(tiles * tiles, ctx->Kc, ch.n);
#define GGF_FL(T, R_, grid, fam, Wp, Pp) \
    flush_kernel<T, R_><<<grid, 256, 0, st>>>(N, fam, (T*)(Wp), (const typename Sc<T>::R*)(Pp), ch.pend, ch.kmax, tiles)
    int nl = 1 + (ctx->Kc ? 1 : 0);
    if (!fp64 && ctx->use_tc) {
        nl = 0;
        GGF_TRY(ggf_flush_tc(ctx, st, &nl));
    } else if (g.r == 4) {
        if (fp64) { GGF_FL(double, 4, gr, ctx->K, ch.Wr, ch.Pr); if (ctx->Kc) GGF_FL(cxd, 4, gc, ctx->Kc, ch.Wc, ch.Pc); }
        else { GGF_FL(float, 4, gr, ctx->K, ch.Wr, ch.Pr); if (ctx->Kc) GGF_FL(cxf, 4, gc, ctx->Kc, ch.Wc, ch.Pc); }
    } else {
        if (fp64) { GGF_FL(double, 8, gr, ctx->K, ch.Wr, ch.Pr); if (ctx->Kc) GGF_FL(cxd, 8, gc, ctx->Kc, ch.Wc, ch.Pc); }
        else { GGF_FL(float, 8, gr, ctx->K, ch.Wr, ch.Pr); if (ctx->Kc) GGF_FL(cxf, 8, gc, ctx->Kc, ch.Wc, ch.Pc); }
    }
#undef GGF_FL
    ctx->prof_pair(GGF_KT_FLUSH, ev0, ctx->prof_mark(st));
    reset_pend<<<(ch.n + 127) / 128, 128, 0, st>>>(ch.n, ch.pend);
    ctx->launches += nl + 1;
    GGF_CK(cudaGetLastError());
    ch.steps_since_flush = 0;
    return GGF_OK;
}

__global__ void bump_sweep(unsigned long long* s) { *s += 1ULL; }

// Kernel attributes are set once per context before any launch, so that no
// attribute call happens while a sweep is being captured into a graph.
// The attribute is a per-function cap shared by every context in the
// process, so it is raised once to the device's opt-in maximum.
ggf_status ggf_prepare_sampler(ggf_ctx* ctx) {
    static bool done[64] = {false};
    if (ctx->device >= 0 && ctx->device < 64 && done[ctx->device]) return GGF_OK;
    int mx = 0;
    GGF_CK(cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    // dynamic cap = opt-in limit minus the kernel's static shared memory
    auto cap = [&](const void* fn) -> ggf_status {
        cudaFuncAttributes fa;
        GGF_CK(cudaFuncGetAttributes(&fa, fn));
        GGF_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, mx - (int)fa.sharedSizeBytes));
        return GGF_OK;
    };
    GGF_TRY(cap((const void*)ratio_kernel<double, cxd, false, 4>));
    GGF_TRY(cap((const void*)ratio_kernel<double, cxd, false, 8>));
    GGF_TRY(cap((const void*)ratio_kernel<float, cxf, false, 4>));
    GGF_TRY(cap((const void*)ratio_kernel<float, cxf, false, 8>));
    GGF_TRY(cap((const void*)ratio_kernel<double, cxd, true, 8>));
    GGF_TRY(cap((const void*)ratio_kernel<float, cxf, true, 8>));
    GGF_TRY(cap((const void*)gather_kernel<double, cxd, 4>));
    GGF_TRY(cap((const void*)gather_kernel<double, cxd, 8>));
    GGF_TRY(cap((const void*)gather_kernel<float, cxf, 4>));
    GGF_TRY(cap((const void*)gather_kernel<float, cxf, 8>));
    if (ctx->device >= 0 && ctx->device < 64) done[ctx->device] = true;
    return GGF_OK;
}

ggf_status ggf_bump_sweep(ggf_ctx* ctx, cudaStream_t st) {
    bump_sweep<<<1, 1, 0, st>>>(ctx->ch.d_sweep);
    ctx->launches += 1;
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}

ggf_status ggf_observe(ggf_ctx* ctx, double* d_obs, cudaStream_t st) {
    Chains& ch = ctx->ch;
    ctx->launches += 1;
    observe_kernel<<<ch.n, 256, 0, st>>>(ctx->dc(), ch.n, ch.links, ch.ell, ch.sweep_acc, d_obs);
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}

ggf_status ggf_mark_refresh(ggf_ctx* ctx, cudaStream_t st) {
    Chains& ch = ctx->ch;
    GGF_CK(cudaMemsetAsync(ch.refresh_list, 0, sizeof(int), st));
    ctx->launches += 1;
    mark_refresh<<<(ch.n + 127) / 128, 128, 0, st>>>(ch.n, ch.opts.refresh_every, ch.since_refresh, ch.refresh_list);
    GGF_CK(cudaGetLastError());
    return GGF_OK;
}
