// Link steps of the batched updates (the batch scheme is in k_batch.cu): for
// every chain, the kb Metropolis proposals of a batch run in order on the
// small matrix W[T, T] of every pair.
//
// One thread-block cluster per chain.  The pairs are dealt to the cluster's
// CTAs (a complex pair counts four real ones), each CTA keeps its pairs'
// matrices, and only the Pfaffian ratios cross CTAs: one cluster barrier per
// proposal, after which every CTA combines the same numbers in the same
// order and so takes the same decision.
//
// Storage: at link j only G[F, F] (F: the later links' rows) and the leading
// block X[0 .. j r, 0 .. j r] are live, so one kr x kr matrix holds both (X
// grows over what G has left), in shared memory where it fits (FP32 up to
// rank 128 for one complex pair), else in the pair's X slot in global memory
// (L2).  G0, needed for P and Q, is the untouched G slot, read one link ahead
// of its use.
//
// What bounds it: the chain of dependent FP64 steps of a proposal (a Pfaffian
// of order 2 r, a solve of order r, the combination).  The FP64 unit takes two
// lanes per clock and SM, so a warp's instruction holds one of the four
// sub-units for 64 cycles, and the tasks of a
// proposal run on different ones: the Pfaffian on a warp, the solve on two
// whether or not the proposal will be accepted, the log-weights one link later
// on another.  What does not depend on the decision runs beside them: P and Q,
// the next link's Delta, the next slices of G0.  Thousand cycles per link of a
// complex pair of rank 128 in FP32: Pfaffian 32 - 39, solve 34 - 48, barrier and
// decision 4, update 14 - 18 (29 on the first link).
// Measured per batch of 16 links, against one CTA per chain that took its
// pairs in turn with G and X in L2: 16 chains of 16 x 16 U(1), K = 4 (rank
// 128) 8.70 -> 0.97 ms (two waves: 15 clusters of 8 fit); 96 chains of 5 x 5
// SU(2), K = 2 (rank 64) 0.92 -> 0.23 ms; 24 FP64 chains of 8 x 8 U(1), K = 2
// (rank 128) 9.7 -> 3.6 ms.  Rolled loops and calls in place of expanded code
// (half the instructions) were 10% slower.
#include <algorithm>
#include <cooperative_groups.h>
#include "ggf_sweep.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int ST = 256;            // threads per CTA
constexpr int SWARPS = ST / 32;

struct StepArgs {
    DevConst dc;
    const unsigned long long* d_sweep;
    int l0, kb, KRM;
    uint64_t seed;
    uint64_t coff;         // Philox key word 1 = coff + chain
    double width;
    void* links;
    cxd* ell;
    int* since_refresh;
    int* sweep_acc;
    unsigned long long* counters;
    int* pend;
    void* Sr;         // small matrices [n][K][2][KRM][KRM]: G0 then X
    void* Sc_;        // [n][Kc][2][KRM][KRM]
    PairBins bins;
    // resident[b]: the matrices of CTA b's pairs live in shared memory; tables[b]: so
    // do every link's Delta and the slices of G0 (else Delta link by link, and
    // the slices read in place)
    unsigned char resident[MAXCS], tables[MAXCS];
};

// Byte offsets of a CTA's shared arrays (host and device compute the same).
struct StepLayout {
    size_t rho, ell, term, prop, tw, task, zs, scratch, pq, g0, delta, mat, total;
    size_t task_bytes;
};

__host__ __device__ inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

// ld of a resident matrix: odd, so that column walks are free of bank conflicts
__host__ __device__ inline int mat_ld(int kr) { return kr + 1; }

// Whether a CTA forms P and Q of every link beside the link's Pfaffian: they do
// not depend on the decision, and the warps that would do it wait otherwise.
// Not for FP64, whose products would take the Pfaffian's unit (and are wasted
// where the proposal is rejected), nor where the pairs' tasks fill the warps.
__host__ __device__ inline bool early_pq(int np, int nc, size_t rw, bool tables) {
    return tables && rw == 4 && (np == 1 || (nc == 0 && np == 2));
}

// Slots for Delta: a CTA that forms P and Q early also forms the next link's
// Delta there, so two do; the doublet rotations of SU(2), four times the
// products, take the whole CTA at the start.
__host__ __device__ inline int delta_slots(bool early, bool tables, bool su2, int kb) {
    return !tables ? 1 : early && !su2 ? 2 : kb;
}

// np pairs, nc of them complex; rw, cw: bytes of a real and a complex element of W
__host__ __device__ inline StepLayout step_layout(int P, int r, int kb, int KRM, int np, int nc, size_t rw, size_t cw,
                                                  bool resident, bool tables, bool su2) {
    StepLayout s;
    const bool early = early_pq(np, nc, rw, tables);
    size_t o = 0;
    auto take = [&](size_t& at, size_t bytes) { at = o; o = up16(o + bytes); };
    take(s.rho, 2 * (size_t)P * sizeof(cxd));
    take(s.ell, (size_t)P * sizeof(cxd));
    take(s.term, (size_t)P * sizeof(cxd));
    take(s.prop, (size_t)kb * sizeof(Proposal));
    take(s.tw, (size_t)kb * 36 * sizeof(double));
    // a task's scratch: W_SS (r x r), the bordered matrix or [A | B] (2r x 2r), a column (r)
    s.task_bytes = (size_t)(5 * r * r + r) * sizeof(cxd);
    take(s.task, (size_t)(2 * np < SWARPS ? 2 * np : SWARPS) * s.task_bytes);
    take(s.zs, (size_t)np * r * r * sizeof(cxd));
    const size_t w = nc ? cw : rw;
    take(s.scratch, (early ? 1 : 3) * (size_t)KRM * r * w);
    take(s.pq, early ? 2 * (size_t)KRM * r * ((np - nc) * rw + nc * cw) : 0);
    take(s.g0, tables ? 2 * (size_t)KRM * r * ((np - nc) * rw + nc * cw) : 0);
    take(s.delta, (size_t)delta_slots(early, tables, su2, kb) * r * r * ((np - nc) * sizeof(double) + nc * sizeof(cxd)));
    take(s.mat, resident ? (size_t)KRM * mat_ld(KRM) * ((np - nc) * rw + nc * cw) : 0);
    s.total = o;
    return s;
}

// Asynchronous copy of BYTES (4, 8 or 16) into shared memory.
template <int BYTES> __device__ __forceinline__ void cp_async(void* dst, const void* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

// One pair's part of link j before the decision: the ratio (task 0) or Z (task 1).
template <class T, int R>
__device__ __forceinline__ void ratio_task(const T* M, int ld, int jr, const typename Fp64Of<T>::Z* D, void* scratch,
                                           cxd* rho_out, int p, int CS) {
    typedef typename Fp64Of<T>::Z Z;
    const int lane = threadIdx.x & 31;
    Z* Ws = (Z*)scratch;
    Z* Bw = Ws + R * R;
    for (int e = lane; e < R * R; e += 32) Ws[e] = wide(M[(size_t)(jr + e / R) * ld + jr + e % R]);
    __syncwarp();
    const Z pf = bordered_ratio(D, Ws, Bw, R);
    if (lane < CS) {
        cxd* dst = rho_out + p;
        if (CS > 1) dst = cg::this_cluster().map_shared_rank(dst, lane);
        *dst = to_c(pf);
    }
    __syncwarp();
}

template <class T, int R>
__device__ __forceinline__ void z_task(const T* M, int ld, int jr, const typename Fp64Of<T>::Z* D, void* scratch,
                                       T* Zout) {
    typedef typename Fp64Of<T>::Z Z;
    const int lane = threadIdx.x & 31;
    Z* Ws = (Z*)scratch;
    Z* Aug = Ws + R * R;          // r x 2r
    Z* Zw = Aug + 2 * R * R;
    Z* fcol = Aug + 4 * R * R;
    for (int e = lane; e < R * R; e += 32) Ws[e] = wide(M[(size_t)(jr + e / R) * ld + jr + e % R]);
    __syncwarp();
    pair_z<sizeof(typename Sc<T>::R) == 4>(D, Ws, Aug, fcol, R, Zw);
    for (int e = lane; e < R * R; e += 32) Zout[e] = narrow(Zw[e], T{});
}

// Z of the CTA's only pair by two warps (the warps w0 and w0 + 1, "part" 0 and
// 1): an FP64 instruction holds one of the SM's four sub-units for 64 cycles
// whatever the number of its lanes, so the products of a step go to two of
// them.  The operations and their order are warp_solve's; rows are exchanged
// while the pivot row is scaled.
template <class T, int R>
__device__ __forceinline__ void z_task_two(const T* M, int ld, int jr, const typename Fp64Of<T>::Z* D, void* scratch,
                                           T* Zout, int part) {
    typedef typename Fp64Of<T>::Z Z;
    typedef ZOps<sizeof(typename Sc<T>::R) == 4> Ops;
    constexpr int W2 = 2 * R;
    const int lane = threadIdx.x & 31, l2 = part * 32 + lane;
    Z* Ws = (Z*)scratch;
    Z* A = Ws + R * R;            // r x 2r
    Z* fcol = A + 4 * R * R;
    auto both = [] { asm volatile("bar.sync 1, 64;" ::: "memory"); };
    for (int e = l2; e < R * R; e += 64) Ws[e] = wide(M[(size_t)(jr + e / R) * ld + jr + e % R]);
    both();
    for (int e = l2; e < R * R; e += 64) {
        const int i = e / R, j = e % R;
        Z v = i == j ? Sc<Z>::one() : Sc<Z>::zero();
#pragma unroll
        for (int z = 0; z < R; ++z) Ops::add(v, D[i * R + z], Ws[z * R + j]);
        A[i * W2 + j] = v;
        A[i * W2 + R + j] = D[e];
    }
    both();
    for (int k = 0; k < R; ++k) {
        const bool in = lane >= k && lane < R;
        const int p = warp_pivot(in ? magc(A[lane * W2 + k]) : 0.0, in);
        const Z d = A[p * W2 + k];
        if (is_zero(d)) break;       // alike in both warps; the ratio is 0 then
        if (part == 0) {
            const Z id = Ops::inv(d);
            if (lane > k && lane < W2) {
                const Z t = A[p * W2 + lane], u = A[k * W2 + lane];
                A[p * W2 + lane] = u;
                A[k * W2 + lane] = Ops::div(t, d, id);
            }
        } else if (lane < R) {
            fcol[lane] = A[(lane == p ? k : lane) * W2 + k];
        }
        both();
        const int j = l2 % W2;
        for (int i = l2 / W2; i < R; i += 64 / W2)
            if (i != k && j > k) Ops::sub(A[i * W2 + j], fcol[i], A[k * W2 + j]);
        both();
    }
    for (int e = l2; e < R * R; e += 64) {
        const Z v = A[(e / R) * W2 + R + e % R];
        Zout[e] = narrow(v, T{});
    }
}

// G := G0 of one pair, a warp per row; asynchronous into shared memory.
template <class T>
__device__ __forceinline__ void copy_g(T* dst, int ld, const T* src, int KRM, int kr, bool shared) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (shared) {
        for (int i = warp; i < kr; i += SWARPS)
            for (int q = lane; q < kr; q += 32) cp_async<sizeof(T)>(dst + (size_t)i * ld + q, src + (size_t)i * KRM + q);
    } else {
        for (int i = warp; i < kr; i += SWARPS)
            for (int q = lane; q < kr; q += 32) dst[(size_t)i * ld + q] = src[(size_t)i * KRM + q];
    }
}

// Slices of G0 that link j needs, into shared memory, both with the R values of
// one index contiguous: G0[a, S] as Gc[a][b] and G0[S, a] as Gr[a][b], a < jr.
template <class T, int R>
__device__ __forceinline__ void g0_fetch(const T* G0, int KRM, int jr, T* Gc, T* Gr) {
    constexpr int E = 16 / sizeof(T);       // elements per copy; R and jr are multiples of it
    for (int e = threadIdx.x; e < jr * (R / E); e += ST) {
        const int a = e / (R / E), b = (e % (R / E)) * E;
        cp_async<16>(Gc + (size_t)a * R + b, G0 + (size_t)a * KRM + jr + b);
    }
    for (int b = threadIdx.x >> 5; b < R; b += SWARPS)
        for (int a = threadIdx.x & 31; a < jr; a += 32)
            cp_async<sizeof(T)>(Gr + (size_t)a * R + b, G0 + (size_t)(jr + b) * KRM + a);
}

// acc -+= x y.  FP32 complex products round as the chains always have: the real
// part's second product and the imaginary part's second product first, each
// then fused with the other, the sum apart (x: the left factor of the row walk).
template <class T> __device__ __forceinline__ void sub_xy(T& r, T x, T y) { acc_sub(r, x, y); }
template <class T> __device__ __forceinline__ void add_xy(T& r, T x, T y) { acc_add(r, x, y); }
__device__ __forceinline__ cxf mul_xy(cxf x, cxf y) {
    return {__fmaf_rn(x.x, y.x, -__fmul_rn(x.y, y.y)), __fmaf_rn(x.y, y.x, __fmul_rn(x.x, y.y))};
}
template <> __device__ __forceinline__ void sub_xy<cxf>(cxf& r, cxf x, cxf y) {
    const cxf t = mul_xy(x, y);
    r = {__fsub_rn(r.x, t.x), __fsub_rn(r.y, t.y)};
}
template <> __device__ __forceinline__ void add_xy<cxf>(cxf& r, cxf x, cxf y) {
    const cxf t = mul_xy(x, y);
    r = {__fadd_rn(r.x, t.x), __fadd_rn(r.y, t.y)};
}

// N contiguous values (16-byte aligned) in 16-byte loads.
template <int N, class T> __device__ __forceinline__ void load_row(T (&v)[N], const T* p) {
    static_assert(N * sizeof(T) % 16 == 0, "whole 16-byte words");
#pragma unroll
    for (int i = 0; i < (int)(N * sizeof(T) / 16); ++i) ((float4*)v)[i] = ((const float4*)p)[i];
}

// P (m x r, m = jr + r): -X G0[0:jr, S] above the identity, and Q (r x m):
// -G0[S, 0:jr] X beside the identity, by nt threads (a multiple of 32) of which
// this is thread t.  A thread keeps the r sums of RB rows (columns): each value
// of X is read once per product, and the reads, which wait in the same queue
// as the FP64 instructions of the Pfaffian beside them, are few per product
// (one row per thread and half of the sums each took twice as long at rank
// 120).  P's rows fill whole warps before Q's columns begin.
// SLICED: the slices of G0 from g0_fetch, else G0 itself.
template <class T, int R, bool SLICED>
__device__ __forceinline__ void pair_pq(const T* M, int ld, int jr, int KRM, const T* Gc, const T* Gr, T* Pm, T* Qm,
                                        int t, int nt) {
    constexpr int RB = sizeof(T) == 4 ? 4 : sizeof(T) == 8 && Sc<T>::CPLX ? 2 : 1;
    constexpr int U = sizeof(T) == 4 ? 32 / R : 2;      // loads in flight where a step has few products
    const int S = (jr + RB - 1) / RB, Sp = (S + 31) & ~31;
    for (int it = t; it < 2 * Sp; it += nt) {
        const bool col = it >= Sp;
        const int a0 = it - (col ? Sp : 0);
        if (a0 >= S) continue;
        const T* x0[RB];
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int a = a0 + k * S < jr ? a0 + k * S : a0;
            x0[k] = M + (col ? (size_t)a : (size_t)a * ld);
        }
        const size_t xs = col ? ld : 1;
        const T* G = col ? Gr : Gc;
        const size_t gq = SLICED ? R : col ? 1 : KRM, gb = SLICED ? 1 : col ? KRM : 1;
        T acc[RB][R];
#pragma unroll
        for (int k = 0; k < RB; ++k)
#pragma unroll
            for (int b = 0; b < R; ++b) acc[k][b] = Sc<T>::zero();
#pragma unroll U
        for (int q = 0; q < jr; ++q) {
            T x[RB];
#pragma unroll
            for (int k = 0; k < RB; ++k) x[k] = x0[k][q * xs];
            if constexpr (SLICED && RB > 1) {
                alignas(16) T gv[R];
                load_row<R>(gv, G + (size_t)q * R);
#pragma unroll
                for (int k = 0; k < RB; ++k)
#pragma unroll
                    for (int b = 0; b < R; ++b) sub_xy(acc[k][b], x[k], gv[b]);
            } else {
#pragma unroll
                for (int b = 0; b < R; ++b) {
                    const T gb_ = G[q * gq + b * gb];
#pragma unroll
                    for (int k = 0; k < RB; ++k) sub_xy(acc[k][b], x[k], gb_);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int a = a0 + k * S;
            if (a < jr) {
#pragma unroll
                for (int b = 0; b < R; ++b) {
                    if (col) Qm[b * KRM + a] = acc[k][b];
                    else Pm[a * R + b] = acc[k][b];
                }
            }
        }
    }
    for (int e = t; e < R * R; e += nt) {
        const int a = e / R, b = e % R;
        Pm[(jr + a) * R + b] = Qm[b * KRM + jr + a] = a == b ? Sc<T>::one() : Sc<T>::zero();
    }
}

// M += left y on n rows and nc columns of M (left: n x R, y: R x nc with row
// length yl): a lane keeps the R values of C columns and walks the rows B at a
// time, whose R values the warp reads as one broadcast for all its columns
// (with one column per lane these reads, a quarter of a warp per cycle, bound
// it).  Rows from zr and columns from zc on start at zero.  Rows and columns
// past the end are computed from the last one and dropped, so that all sums
// interleave.
template <class T, int R, int B, int C>
__device__ __forceinline__ void rank_r_cols(T* M, int ld, const T* left, const T* y, int yl, int n, int nc, int zr, int zc,
                                            int c0) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T yv[R][C];
    int col[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        col[c] = min(c0 + 32 * c + lane, nc - 1);
#pragma unroll
        for (int b = 0; b < R; ++b) yv[b][c] = y[(size_t)b * yl + col[c]];
    }
    for (int i = warp; i < n; i += B * SWARPS) {
        T v[B][C];
        int at[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            at[k] = min(i + k * SWARPS, n - 1);
#pragma unroll
            for (int c = 0; c < C; ++c)
                v[k][c] = at[k] < zr && col[c] < zc ? M[(size_t)at[k] * ld + col[c]] : Sc<T>::zero();
        }
        constexpr int H = B > 1 ? 16 / sizeof(T) : 1;       // values of a left row per load
#pragma unroll
        for (int b = 0; b < R; b += H) {
#pragma unroll
            for (int k = 0; k < B; ++k) {
                alignas(16) T x[H];
                if constexpr (B > 1) load_row<H>(x, left + at[k] * R + b);
                else x[0] = left[at[k] * R + b];
#pragma unroll
                for (int h = 0; h < H; ++h)
#pragma unroll
                    for (int c = 0; c < C; ++c) add_xy(v[k][c], x[h], yv[b + h][c]);
            }
        }
#pragma unroll
        for (int k = 0; k < B; ++k)
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (i + k * SWARPS < n && c0 + 32 * c + lane < nc) M[(size_t)at[k] * ld + col[c]] = v[k][c];
    }
}
template <class T, int R>
__device__ __forceinline__ void rank_r(T* M, int ld, const T* left, const T* y, int yl, int n, int nc, int zr, int zc) {
    if constexpr (sizeof(typename Sc<T>::R) == 8) {         // bound by the FP64 unit
        for (int c0 = 0; c0 < nc; c0 += 32) rank_r_cols<T, R, 1, 1>(M, ld, left, y, yl, n, nc, zr, zc, c0);
    } else {
        int c0 = 0;
        for (; c0 + 32 < nc; c0 += 64) rank_r_cols<T, R, 2, 2>(M, ld, left, y, yl, n, nc, zr, zc, c0);
        if (c0 < nc) rank_r_cols<T, R, 2, 1>(M, ld, left, y, yl, n, nc, zr, zc, c0);
    }
}

// Rank-r update of one pair's matrix after link j was accepted (all threads).
// M: G on the rows and columns >= jr, X on those < jr; afterwards X reaches
// to m = jr + r.  Every element's sum runs over the same terms in the same
// order whichever thread forms it.  ready: P and Q are there already.
template <class T, int R>
__device__ __forceinline__ void pair_update(T* M, int ld, int jr, int kr, int KRM, const T* Zs, const T* Gc,
                                            const T* Gr, bool sliced, T* st, T* Pm, T* Qm, bool ready) {
    const int m = jr + R, nf = kr - m;
    T* A1 = st;                    // -G[F, S] Z (nf x r)
    T* T1 = A1 + (size_t)nf * R;   // P Z (m x r); nf + m = kr
    if (!ready) {
        if (sliced) pair_pq<T, R, true>(M, ld, jr, KRM, Gc, Gr, Pm, Qm, threadIdx.x, ST);
        else pair_pq<T, R, false>(M, ld, jr, KRM, Gc, Gr, Pm, Qm, threadIdx.x, ST);
    }
    for (int e = threadIdx.x; e < nf * R; e += ST) {
        const int i = e / R, b = e - i * R;
        T acc = Sc<T>::zero();
#pragma unroll
        for (int a = 0; a < R; ++a) add_xy(acc, M[(size_t)(m + i) * ld + jr + a], Zs[a * R + b]);
        A1[e] = -acc;
    }
    auto form_t1 = [&] {
        for (int e = threadIdx.x; e < m * R; e += ST) {
            const int a = e / R, b = e - a * R;
            T acc = Sc<T>::zero();
#pragma unroll
            for (int q = 0; q < R; ++q) add_xy(acc, Pm[a * R + q], Zs[q * R + b]);
            T1[e] = acc;
        }
    };
    if (ready) form_t1();
    __syncthreads();
    // G[F, F] -= (G[F, S] Z) G[S, F]: the sign is A1's, which changes no rounding
    if (nf > 0) rank_r<T, R>(M + (size_t)m * ld + m, ld, A1, M + (size_t)jr * ld + m, ld, nf, nf, nf, nf);
    if (!ready) {
        form_t1();
        __syncthreads();
    }
    // X += (P Z) Q on the leading m x m block; rows and columns >= jr start at
    // zero (they held G, of which only columns >= m are still read)
    rank_r<T, R>(M, ld, T1, Qm, KRM, m, m, jr, jr);
    __syncthreads();
}

// SU2: SU(2) links (quaternion proposal and doublet twist); the Z2 and U(1)
// instantiations (SU2 = false) do not contain that code.
template <class RW, class CW, bool SU2, int R>
__global__ void __launch_bounds__(ST, 2) batch_steps(StepArgs a) {
    extern __shared__ __align__(16) unsigned char sm[];
    const Geometry& g = a.dc.g;
    const int P = a.dc.P, K = a.dc.K, Kc = P - K, KRM = a.KRM, kb = a.kb, kr = kb * R;
    const int CS = cg::this_cluster().num_blocks(), rank = cg::this_cluster().block_rank();
    const int c = blockIdx.x / CS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p0 = a.bins.first[rank], np = a.bins.first[rank + 1] - p0;
    int nc = 0;
    for (int s = 0; s < np; ++s) nc += a.bins.ord[p0 + s] >= K;
    const bool resident = a.resident[rank], tables = a.tables[rank];
    const StepLayout lay = step_layout(P, R, kb, KRM, np, nc, sizeof(RW), sizeof(CW), resident, tables, SU2);
    const bool early = early_pq(np, nc, sizeof(RW), tables);
    const int kbt = delta_slots(early, tables, SU2, kb);
    const bool ahead = early && !SU2;       // Delta one link ahead
    cxd* rho = (cxd*)(sm + lay.rho);        // [2][P], by the link's parity
    cxd* ells = (cxd*)(sm + lay.ell);       // [P]
    cxd* term = (cxd*)(sm + lay.term);      // [P] scaled pair terms before the proposal
    Proposal* props = (Proposal*)(sm + lay.prop);
    double* tws = (double*)(sm + lay.tw);   // [kb][36]
    cxd* Zs = (cxd*)(sm + lay.zs);          // [np][R][R]
    __shared__ int s_accept;
    __shared__ unsigned long long s_mask;
    const size_t SS = (size_t)KRM * KRM;
    const int ldr = resident ? mat_ld(KRM) : KRM;

    // the CTA's real pairs come before its complex ones (nr of them)
    const int nr = np - nc;
    auto g0_real = [&](int s) { return (RW*)a.Sr + ((size_t)c * K + a.bins.ord[p0 + s]) * 2 * SS; };
    auto g0_cplx = [&](int s) { return (CW*)a.Sc_ + ((size_t)c * Kc + (a.bins.ord[p0 + s] - K)) * 2 * SS; };
    auto mat_real = [&](int s) {
        return resident ? (RW*)(sm + lay.mat) + (size_t)s * KRM * ldr : g0_real(s) + SS;
    };
    auto mat_cplx = [&](int s) {
        return resident ? (CW*)(sm + lay.mat + (size_t)nr * KRM * ldr * sizeof(RW)) + (size_t)(s - nr) * KRM * ldr
                        : g0_cplx(s) + SS;
    };
    auto del_real = [&](int s) { return (double*)(sm + lay.delta) + (size_t)s * kbt * R * R; };
    auto del_cplx = [&](int s) {
        return (cxd*)(sm + lay.delta + (size_t)nr * kbt * R * R * sizeof(double)) + (size_t)(s - nr) * kbt * R * R;
    };
    // P and Q of a pair: its own where they are formed early, else shared
    auto pm_real = [&](int s) { return early ? (RW*)(sm + lay.pq) + (size_t)s * 2 * KRM * R : (RW*)(sm + lay.scratch) + (size_t)KRM * R; };
    auto pm_cplx = [&](int s) {
        return early ? (CW*)(sm + lay.pq + (size_t)nr * 2 * KRM * R * sizeof(RW)) + (size_t)(s - nr) * 2 * KRM * R
                     : (CW*)(sm + lay.scratch) + (size_t)KRM * R;
    };
    auto sl_real = [&](int s) { return (RW*)(sm + lay.g0) + (size_t)s * 2 * KRM * R; };
    auto sl_cplx = [&](int s) {
        return (CW*)(sm + lay.g0 + (size_t)nr * 2 * KRM * R * sizeof(RW)) + (size_t)(s - nr) * 2 * KRM * R;
    };

    // ---- everything that no decision of the batch changes
    for (int s = 0; s < np; ++s) {
        // G := G0, in flight while the proposals are drawn
        if (s < nr) copy_g<RW>(mat_real(s), ldr, g0_real(s), KRM, kr, resident);
        else copy_g<CW>(mat_cplx(s), ldr, g0_cplx(s), KRM, kr, resident);
    }
    if (threadIdx.x == 0) s_mask = 0;
    const unsigned long long sweep = *a.d_sweep;
    for (int j = threadIdx.x; j < kb; j += ST) {
        double* tw = tws + j * 36;
        if constexpr (SU2) {
            Proposal q{};
            q.u_acc = draw_su2(g, a.links, c, a.l0 + j, sweep, a.seed, a.width, tw, tw + 4, tw + 20, a.coff);
            props[j] = q;
        } else {
            props[j] = draw_proposal(g, a.links, c, a.l0 + j, sweep, a.seed, a.width, a.coff);
        }
    }
    for (int p = threadIdx.x; p < P; p += ST) ells[p] = a.ell[(size_t)c * P + p];
    __syncthreads();
    if constexpr (!SU2)
        if (g.group == GGF_U1) {
            // the twists, one sine and cosine per thread
            for (int e = threadIdx.x; e < kb * 2 * g.n_v; e += ST) {
                const int j = e / (2 * g.n_v), t = e % (2 * g.n_v), md = t % g.n_v, nw = t / g.n_v;
                double sv, cv;
                sincos(g.q[md] * (nw ? props[j].th_new : props[j].th_old), &sv, &cv);
                tws[j * 36 + 4 * nw + 2 * md] = cv;
                tws[j * 36 + 4 * nw + 2 * md + 1] = sv;
            }
            __syncthreads();
        }
    // Delta of link j into slot d, by nt threads of which this is thread t
    auto fill_delta = [&](int j, int d, int t, int nt) {
        for (int s = 0; s < np; ++s) {
            const int p = a.bins.ord[p0 + s];
            for (int x = t; x < R * R; x += nt) {
                const int e = d * R * R + x;
                if (s < nr) del_real(s)[e] = delta_elem<double>(a.dc, p, a.l0 + j, x / R, x % R, props[j], tws + j * 36, SU2);
                else del_cplx(s)[e] = delta_elem<cxd>(a.dc, p - K, a.l0 + j, x / R, x % R, props[j], tws + j * 36, SU2);
            }
        }
    };
    if (ahead) fill_delta(0, 0, threadIdx.x, ST);
    else if (tables)
        for (int e = threadIdx.x / (R * R); e < kb; e += ST / (R * R)) fill_delta(e, e, threadIdx.x % (R * R), R * R);
    asm volatile("cp.async.wait_all;" ::: "memory");
    // every CTA of the cluster is running before the first remote write
    if (CS > 1) cg::this_cluster().sync();
    else __syncthreads();

    auto fetch = [&](int jr) {
        for (int s = 0; s < np && tables && jr > 0; ++s) {
            if (s < nr) g0_fetch<RW, R>(g0_real(s), KRM, jr, sl_real(s), sl_real(s) + (size_t)KRM * R);
            else g0_fetch<CW, R>(g0_cplx(s), KRM, jr, sl_cplx(s), sl_cplx(s) + (size_t)KRM * R);
        }
    };
    const bool two = np == 1 && R == 8;     // a block of order 4 is too small for two warps
    const int tw_tasks = two ? 3 : 2 * np;  // warps with a task; early: the next ones form P and Q
    int prev = 0;                       // the previous link was accepted
    for (int j = 0; j < kb; ++j) {
        const int jr = j * R;
        cxd* rj = rho + (j & 1) * P;
        if (!tables) {
            fill_delta(j, 0, threadIdx.x, ST);
            __syncthreads();
        }
        const int dj = ahead ? j & 1 : tables ? j : 0;
        if (!early) fetch(jr);
        if (warp == SWARPS - 1) {
            // log-weights after the previous link, then the scaled pair terms
            const cxd* rp = rho + ((j & 1) ^ 1) * P;
            double amax = -INFINITY;
            for (int p = lane; p < P; p += 32) {
                if (prev) ell_add(ells[p], rp[p], p < K);
                amax = fmax(amax, a.dc.logc[p].x + ells[p].x);
            }
            for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            for (int p = lane; p < P; p += 32) {
                cxd e = a.dc.logc[p] + ells[p];
                e.x -= amax;
                term[p] = a.dc.w[p] * (p < K ? cxd{exp(e.x), 0.0} : cexp_(e));
            }
        }
        // Delta of the next link: after the log-weights, or by the last of the warps
        // for P and Q where the log-weights take longer than the Pfaffian
        if (ahead && j + 1 < kb && warp == SWARPS - (nc && R == 8 ? 1 : 2)) fill_delta(j + 1, (j + 1) & 1, lane, 32);
        if (early && warp >= tw_tasks && warp < SWARPS - 1) {
            const int t = threadIdx.x - 32 * tw_tasks, nt = 32 * (SWARPS - 1 - tw_tasks);
            for (int s = 0; s < np; ++s) {
                if (s < nr)
                    pair_pq<RW, R, true>(mat_real(s), ldr, jr, KRM, sl_real(s), sl_real(s) + (size_t)KRM * R, pm_real(s),
                                         pm_real(s) + (size_t)KRM * R, t, nt);
                else
                    pair_pq<CW, R, true>(mat_cplx(s), ldr, jr, KRM, sl_cplx(s), sl_cplx(s) + (size_t)KRM * R, pm_cplx(s),
                                         pm_cplx(s) + (size_t)KRM * R, t, nt);
            }
        }
        for (int t = warp; t < (two ? 3 : 2 * np); t += SWARPS) {
            const int s = two ? 0 : t >> 1, p = a.bins.ord[p0 + s];
            const int kind = two ? (t > 0) : (t & 1);
            void* scr = sm + lay.task + (size_t)(two ? kind : warp) * lay.task_bytes;
            if (s < nr) {
                const double* D = del_real(s) + dj * R * R;
                if (!kind) ratio_task<RW, R>(mat_real(s), ldr, jr, D, scr, rj, p, CS);
                else if (two) z_task_two<RW, R>(mat_real(s), ldr, jr, D, scr, (RW*)Zs, t - 1);
                else z_task<RW, R>(mat_real(s), ldr, jr, D, scr, (RW*)(Zs + s * R * R));
            } else {
                const cxd* D = del_cplx(s) + dj * R * R;
                if (!kind) ratio_task<CW, R>(mat_cplx(s), ldr, jr, D, scr, rj, p, CS);
                else if (two) z_task_two<CW, R>(mat_cplx(s), ldr, jr, D, scr, (CW*)Zs, t - 1);
                else z_task<CW, R>(mat_cplx(s), ldr, jr, D, scr, (CW*)(Zs + s * R * R));
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (CS > 1) cg::this_cluster().sync();
        else __syncthreads();
        if (warp == 0) {
            double so = 0.0, sn = 0.0;
            for (int p = lane; p < P; p += 32) {
                so += term[p].x;
                sn += (term[p] * rj[p]).x;
            }
            for (int o = 16; o > 0; o >>= 1) {
                so += __shfl_xor_sync(0xffffffffu, so, o);
                sn += __shfl_xor_sync(0xffffffffu, sn, o);
            }
            if (lane == 0) {
                const int acc = (sn > 0.0 && so > 0.0 && props[j].u_acc < sn / so) ? 1 : 0;
                s_accept = acc;
                if (acc) s_mask |= 1ULL << j;
            }
        }
        __syncthreads();
        prev = s_accept;
        if (early && j + 1 < kb) fetch(jr + R);     // the slices of link j are done with
        if (prev) {
            for (int s = 0; s < np; ++s) {
                if (s < nr)
                    pair_update<RW, R>(mat_real(s), ldr, jr, kr, KRM, (const RW*)(Zs + s * R * R),
                                       tables ? sl_real(s) : g0_real(s) + jr,
                                       tables ? sl_real(s) + (size_t)KRM * R : g0_real(s) + (size_t)jr * KRM, tables,
                                       (RW*)(sm + lay.scratch), pm_real(s), pm_real(s) + (size_t)KRM * R, early);
                else
                    pair_update<CW, R>(mat_cplx(s), ldr, jr, kr, KRM, (const CW*)(Zs + s * R * R),
                                       tables ? sl_cplx(s) : g0_cplx(s) + jr,
                                       tables ? sl_cplx(s) + (size_t)KRM * R : g0_cplx(s) + (size_t)jr * KRM, tables,
                                       (CW*)(sm + lay.scratch), pm_cplx(s), pm_cplx(s) + (size_t)KRM * R, early);
            }
        } else {
            // rejected: the rows and columns of S belong to X from here on, as zeros
            const int m = jr + R;
            for (int s = 0; s < np; ++s)
                for (int e = threadIdx.x; e < m * R; e += ST) {
                    const int i = e / R, b = jr + e % R;
                    if (s < nr) mat_real(s)[(size_t)i * ldr + b] = mat_real(s)[(size_t)b * ldr + i] = Sc<RW>::zero();
                    else mat_cplx(s)[(size_t)i * ldr + b] = mat_cplx(s)[(size_t)b * ldr + i] = Sc<CW>::zero();
                }
            __syncthreads();
        }
        if (early) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
        }
    }
    // ---- results: X of the CTA's pairs; links, log-weights and counts by rank 0
    if (resident)
        for (int s = 0; s < np; ++s) {
            if (s < nr) {
                const RW* src = mat_real(s);
                RW* dst = g0_real(s) + SS;
                for (int i = warp; i < kr; i += SWARPS)
                    for (int q = lane; q < kr; q += 32) dst[(size_t)i * KRM + q] = src[(size_t)i * ldr + q];
            } else {
                const CW* src = mat_cplx(s);
                CW* dst = g0_cplx(s) + SS;
                for (int i = warp; i < kr; i += SWARPS)
                    for (int q = lane; q < kr; q += 32) dst[(size_t)i * KRM + q] = src[(size_t)i * ldr + q];
            }
        }
    if (rank != 0) return;
    const unsigned long long mask = s_mask;
    for (int p = threadIdx.x; p < P; p += ST) {
        cxd e = ells[p];
        if (prev) ell_add(e, rho[((kb - 1) & 1) * P + p], p < K);
        a.ell[(size_t)c * P + p] = e;
    }
    for (int j = threadIdx.x; j < kb; j += ST) {
        if (!((mask >> j) & 1)) continue;
        const size_t at = (size_t)c * g.n_links + a.l0 + j;
        if constexpr (SU2) {
            for (int k = 0; k < 4; ++k) ((double*)a.links)[at * 4 + k] = tws[j * 36 + k];
        } else {
            if (g.group == GGF_Z2) ((int8_t*)a.links)[at] = (int8_t)props[j].g_new;
            else ((double*)a.links)[at] = props[j].th_new;
        }
    }
    if (threadIdx.x == 0) {
        const int acc = __popcll(mask);
        atomicAdd(&a.counters[0], (unsigned long long)kb);
        if (acc) {
            atomicAdd(&a.counters[1], (unsigned long long)acc);
            a.since_refresh[c] += acc;
            a.sweep_acc[c] += acc;
        }
        a.pend[c] = acc ? kb : 0;
    }
}

// Bins of the pairs (deal_pairs), and for each CTA how much of its data fits in
// shared memory.  Returns the CTAs and the shared memory of the largest.
int step_bins(int K, int Kc, int r, int kb, int KRM, size_t rw, size_t cw, bool su2, size_t smem_max, StepArgs& a,
              size_t& smem) {
    const int CS = deal_pairs(K, Kc, a.bins);
    smem = 0;
    for (int b = 0; b < CS; ++b) {
        const int np = a.bins.first[b + 1] - a.bins.first[b];
        int nc = 0;
        for (int s = 0; s < np; ++s) nc += a.bins.ord[a.bins.first[b] + s] >= K;
        size_t need = 0;
        for (int level = 0; level < 3; ++level) {
            a.resident[b] = level == 0;
            a.tables[b] = level < 2;
            need = step_layout(K + Kc, r, kb, KRM, np, nc, rw, cw, level == 0, level < 2, su2).total;
            if (need <= smem_max) break;
        }
        smem = std::max(smem, need);
    }
    return CS;
}

template <class F> void for_each_step_kernel(F f) {
    f((const void*)batch_steps<double, cxd, false, 4>);
    f((const void*)batch_steps<double, cxd, false, 8>);
    f((const void*)batch_steps<float, cxf, false, 4>);
    f((const void*)batch_steps<float, cxf, false, 8>);
    f((const void*)batch_steps<double, cxd, true, 8>);
    f((const void*)batch_steps<float, cxf, true, 8>);
}

constexpr size_t STEP_STATIC = 256;     // the kernel's static shared variables

size_t step_smem_max(ggf_ctx* ctx) {
    int mx = 0;
    cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
    return (size_t)mx - STEP_STATIC;
}

}  // namespace

ggf_status ggf_prepare_steps(ggf_ctx* ctx) {
    ggf_status rc = GGF_OK;
    for_each_step_kernel([&](const void* fn) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)step_smem_max(ctx));
        if (e != cudaSuccess && rc == GGF_OK) rc = ggf_cuda(ctx, e, "cudaFuncSetAttribute(batch_steps)");
    });
    return rc;
}

// Whether the link steps of batches of kmax links fit the device's shared memory.
bool ggf_steps_fit(ggf_ctx* ctx, int kmax, bool fp64) {
    StepArgs a;
    size_t smem = 0;
    const size_t mx = step_smem_max(ctx);
    step_bins(ctx->K, ctx->Kc, ctx->g.r, kmax, kmax * ctx->g.r, fp64 ? 8 : 4, fp64 ? 16 : 8,
              ctx->g.group == GGF_SU2, mx, a, smem);
    return smem <= mx;
}

// Link steps l0 .. l0 + kb - 1 of every chain on the small matrices Sr, Sc_.
ggf_status ggf_batch_steps(ggf_ctx* ctx, int l0, int kb, void* Sr, void* Sc_, cudaStream_t st) {
    Chains& ch = ctx->ch;
    const Geometry& g = ctx->g;
    const bool fp64 = ch.opts.precision == GGF_FP64;
    StepArgs a;
    a.dc = ctx->dc();
    a.d_sweep = ch.d_sweep;
    a.l0 = l0;
    a.kb = kb;
    a.KRM = ch.kmax * g.r;
    a.seed = ch.opts.seed;
    a.coff = ch.opts.chain_offset;
    a.width = ch.opts.width;
    a.links = ch.links;
    a.ell = ch.ell;
    a.since_refresh = ch.since_refresh;
    a.sweep_acc = ch.sweep_acc;
    a.counters = ch.counters;
    a.pend = ch.pend;
    a.Sr = Sr;
    a.Sc_ = Sc_;
    size_t smem = 0;
    const int CS = step_bins(ctx->K, ctx->Kc, g.r, kb, a.KRM, fp64 ? 8 : 4, fp64 ? 16 : 8, g.group == GGF_SU2,
                             step_smem_max(ctx), a, smem);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ch.n * CS);
    cfg.blockDim = dim3(ST);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CS > 1 ? 1 : 0;
    if (g.group == GGF_SU2) {
        if (fp64) GGF_CK(cudaLaunchKernelEx(&cfg, batch_steps<double, cxd, true, 8>, a));
        else GGF_CK(cudaLaunchKernelEx(&cfg, batch_steps<float, cxf, true, 8>, a));
    } else if (g.r == 4) {
        if (fp64) GGF_CK(cudaLaunchKernelEx(&cfg, batch_steps<double, cxd, false, 4>, a));
        else GGF_CK(cudaLaunchKernelEx(&cfg, batch_steps<float, cxf, false, 4>, a));
    } else {
        if (fp64) GGF_CK(cudaLaunchKernelEx(&cfg, batch_steps<double, cxd, false, 8>, a));
        else GGF_CK(cudaLaunchKernelEx(&cfg, batch_steps<float, cxf, false, 8>, a));
    }
    return GGF_OK;
}
