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
// of order 2 r, a solve of order r, the combination); everything that does not
// depend on the previous decision (random numbers, twists, the changes Delta
// of all kb links) is computed at the start, the solve runs beside the
// Pfaffian whether or not the proposal will be accepted, and the log-weights
// follow one link later, beside the next Pfaffian.
// Measured per batch of 16 links, against one CTA per chain that took its
// pairs in turn with G and X in L2: 16 chains of 16 x 16 U(1), K = 4 (rank
// 128) 8.70 -> 1.23 ms; 96 chains of 5 x 5 SU(2), K = 2 (rank 64) 0.92 -> 0.25
// ms; 24 FP64 chains of 8 x 8 U(1), K = 2 (rank 128) 9.7 -> 3.6 ms.
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
    size_t rho, ell, term, prop, tw, task, zs, scratch, g0, delta, mat, total;
    size_t task_bytes;
};

__host__ __device__ inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

// ld of a resident matrix: odd, so that column walks are free of bank conflicts
__host__ __device__ inline int mat_ld(int kr) { return kr + 1; }

// np pairs, nc of them complex; rw, cw: bytes of a real and a complex element of W
__host__ __device__ inline StepLayout step_layout(int P, int r, int kb, int KRM, int np, int nc, size_t rw, size_t cw,
                                                  bool resident, bool tables) {
    StepLayout s;
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
    take(s.scratch, 3 * (size_t)KRM * r * w);
    take(s.g0, tables ? 2 * (size_t)KRM * r * ((np - nc) * rw + nc * cw) : 0);
    take(s.delta, (size_t)(tables ? kb : 1) * r * r * ((np - nc) * sizeof(double) + nc * sizeof(cxd)));
    take(s.mat, resident ? (size_t)KRM * mat_ld(KRM) * ((np - nc) * rw + nc * cw) : 0);
    s.total = o;
    return s;
}

__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
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
    pair_z(D, Ws, Aug, fcol, R, Zw);
    for (int e = lane; e < R * R; e += 32) Zout[e] = narrow(Zw[e], T{});
}

// Slices of G0 that link j needs, into shared memory: column block G0[0 .. jr, S]
// as Gc[a][b] and row block G0[S, 0 .. jr] as Gr[b][a] (row length KRM).
template <class T, int R>
__device__ __forceinline__ void g0_fetch(const T* G0, int KRM, int jr, T* Gc, T* Gr) {
    constexpr int E = 16 / sizeof(T);       // elements per copy; R and jr are multiples of it
    for (int e = threadIdx.x; e < jr * (R / E); e += ST) {
        const int a = e / (R / E), b = (e % (R / E)) * E;
        cp16(Gc + (size_t)a * R + b, G0 + (size_t)a * KRM + jr + b);
    }
    const int cols = jr / E;
    for (int e = threadIdx.x; e < R * cols; e += ST) {
        const int b = e / cols, a = (e % cols) * E;
        cp16(Gr + (size_t)b * KRM + a, G0 + (size_t)(jr + b) * KRM + a);
    }
}

// Rank-r update of one pair's matrix after link j was accepted (all threads).
// M: G on the rows and columns >= jr, X on those < jr; afterwards X reaches
// to m = jr + r.  Every element's sum runs over the same terms in the same
// order whichever thread forms it.
template <class T, int R>
__device__ __forceinline__ void pair_update(T* M, int ld, int jr, int kr, int KRM, const T* Zs, const T* Gc,
                                            int gcs, const T* Gr, T* st) {
    const int m = jr + R, nf = kr - m;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T* A1 = st;                    // G[F, S] Z (nf x r)
    T* T1 = A1 + (size_t)nf * R;   // P Z (m x r); nf + m = kr
    T* Pm = st + (size_t)KRM * R;  // P (m x r): -X G0[0:jr, S] above the identity
    T* Qm = Pm + (size_t)KRM * R;  // Q (r x m): -G0[S, 0:jr] X beside the identity
    const T one = Sc<T>::one();
    // half the CTA walks rows of X for P, the other half columns for Q: one
    // thread keeps a row's (column's) r sums in registers, so that every
    // element of X is read once per product
    if (threadIdx.x < ST / 2) {
        for (int a = threadIdx.x; a < m; a += ST / 2) {
            T acc[R];
#pragma unroll
            for (int b = 0; b < R; ++b) acc[b] = Sc<T>::zero();
            if (a < jr) {
                const T* xr = M + (size_t)a * ld;
#pragma unroll 2
                for (int q = 0; q < jr; ++q) {
                    const T x = xr[q];
#pragma unroll
                    for (int b = 0; b < R; ++b) acc_sub(acc[b], x, Gc[(size_t)q * gcs + b]);
                }
            }
#pragma unroll
            for (int b = 0; b < R; ++b) Pm[a * R + b] = (a >= jr && b == a - jr) ? one : acc[b];
        }
    } else {
        for (int cc = threadIdx.x - ST / 2; cc < m; cc += ST / 2) {
            T acc[R];
#pragma unroll
            for (int b = 0; b < R; ++b) acc[b] = Sc<T>::zero();
            if (cc < jr) {
#pragma unroll 2
                for (int q = 0; q < jr; ++q) {
                    const T x = M[(size_t)q * ld + cc];
#pragma unroll
                    for (int b = 0; b < R; ++b) acc_sub(acc[b], Gr[(size_t)b * KRM + q], x);
                }
            }
#pragma unroll
            for (int b = 0; b < R; ++b) Qm[b * KRM + cc] = (cc >= jr && b == cc - jr) ? one : acc[b];
        }
    }
    for (int e = threadIdx.x; e < nf * R; e += ST) {
        const int i = e / R, b = e - i * R;
        T acc = Sc<T>::zero();
#pragma unroll
        for (int a = 0; a < R; ++a) acc_add(acc, M[(size_t)(m + i) * ld + jr + a], Zs[a * R + b]);
        A1[e] = acc;
    }
    __syncthreads();
    // G[F, F] -= (G[F, S] Z) G[S, F]: a lane keeps its column's r values and
    // walks the rows, whose r values the warp reads as one broadcast
    for (int j0 = 0; j0 < nf; j0 += 32) {
        const int jj = j0 + lane;
        T y[R];
#pragma unroll
        for (int b = 0; b < R; ++b) y[b] = jj < nf ? M[(size_t)(jr + b) * ld + m + jj] : Sc<T>::zero();
        for (int i = warp; i < nf; i += SWARPS) {
            T* gp = M + (size_t)(m + i) * ld + m + jj;
            if (jj < nf) {
                T acc = *gp;
#pragma unroll
                for (int b = 0; b < R; ++b) acc_sub(acc, A1[i * R + b], y[b]);
                *gp = acc;
            }
        }
    }
    for (int e = threadIdx.x; e < m * R; e += ST) {
        const int a = e / R, b = e - a * R;
        T acc = Sc<T>::zero();
#pragma unroll
        for (int q = 0; q < R; ++q) acc_add(acc, Pm[a * R + q], Zs[q * R + b]);
        T1[e] = acc;
    }
    __syncthreads();
    // X += (P Z) Q on the leading m x m block; rows and columns >= jr start at
    // zero (they held G)
    for (int c0 = 0; c0 < m; c0 += 32) {
        const int cc = c0 + lane;
        T y[R];
#pragma unroll
        for (int b = 0; b < R; ++b) y[b] = cc < m ? Qm[b * KRM + cc] : Sc<T>::zero();
        for (int a = warp; a < m; a += SWARPS) {
            T* xp = M + (size_t)a * ld + cc;
            if (cc < m) {
                T acc = (a < jr && cc < jr) ? *xp : Sc<T>::zero();
#pragma unroll
                for (int b = 0; b < R; ++b) acc_add(acc, T1[a * R + b], y[b]);
                *xp = acc;
            }
        }
    }
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
    const StepLayout lay = step_layout(P, R, kb, KRM, np, nc, sizeof(RW), sizeof(CW), resident, tables);
    const int kbt = tables ? kb : 1;
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
    auto sl_real = [&](int s) { return (RW*)(sm + lay.g0) + (size_t)s * 2 * KRM * R; };
    auto sl_cplx = [&](int s) {
        return (CW*)(sm + lay.g0 + (size_t)nr * 2 * KRM * R * sizeof(RW)) + (size_t)(s - nr) * 2 * KRM * R;
    };

    // ---- everything that no decision of the batch changes
    if (threadIdx.x == 0) s_mask = 0;
    const unsigned long long sweep = *a.d_sweep;
    for (int j = threadIdx.x; j < kb; j += ST) {
        double* tw = tws + j * 36;
        if constexpr (SU2) {
            Proposal q{};
            q.u_acc = draw_su2(g, a.links, c, a.l0 + j, sweep, a.seed, a.width, tw, tw + 4, tw + 20, a.coff);
            props[j] = q;
        } else {
            const Proposal q = draw_proposal(g, a.links, c, a.l0 + j, sweep, a.seed, a.width, a.coff);
            props[j] = q;
            if (g.group == GGF_U1)
                for (int t = 0; t < 2 * g.n_v; ++t) {
                    const int md = t % g.n_v, nw = t / g.n_v;
                    double sv, cv;
                    sincos(g.q[md] * (nw ? q.th_new : q.th_old), &sv, &cv);
                    tw[4 * nw + 2 * md] = cv;
                    tw[4 * nw + 2 * md + 1] = sv;
                }
        }
    }
    for (int p = threadIdx.x; p < P; p += ST) ells[p] = a.ell[(size_t)c * P + p];
    for (int s = 0; s < np; ++s) {
        // G := G0 (row walks of the G slot, coalesced)
        if (s < nr) {
            const RW* src = g0_real(s);
            RW* dst = mat_real(s);
            for (int i = warp; i < kr; i += SWARPS)
                for (int q = lane; q < kr; q += 32) dst[(size_t)i * ldr + q] = src[(size_t)i * KRM + q];
        } else {
            const CW* src = g0_cplx(s);
            CW* dst = mat_cplx(s);
            for (int i = warp; i < kr; i += SWARPS)
                for (int q = lane; q < kr; q += 32) dst[(size_t)i * ldr + q] = src[(size_t)i * KRM + q];
        }
    }
    __syncthreads();
    // Delta of the links j0 .. j0 + kbt - 1
    auto fill_delta = [&](int j0) {
        for (int s = 0; s < np; ++s) {
            const int p = a.bins.ord[p0 + s];
            for (int e = threadIdx.x; e < kbt * R * R; e += ST) {
                const int j = j0 + e / (R * R), x = e % (R * R);
                if (s < nr) del_real(s)[e] = delta_elem<double>(a.dc, p, a.l0 + j, x / R, x % R, props[j], tws + j * 36, SU2);
                else del_cplx(s)[e] = delta_elem<cxd>(a.dc, p - K, a.l0 + j, x / R, x % R, props[j], tws + j * 36, SU2);
            }
        }
    };
    if (tables) fill_delta(0);
    // every CTA of the cluster is running before the first remote write
    if (CS > 1) cg::this_cluster().sync();
    else __syncthreads();

    int prev = 0;                       // the previous link was accepted
    for (int j = 0; j < kb; ++j) {
        const int jr = j * R;
        cxd* rj = rho + (j & 1) * P;
        if (!tables) {
            fill_delta(j);
            __syncthreads();
        }
        const int dj = tables ? j : 0;
        for (int s = 0; s < np && tables && j > 0; ++s) {
            if (s < nr) g0_fetch<RW, R>(g0_real(s), KRM, jr, sl_real(s), sl_real(s) + (size_t)KRM * R);
            else g0_fetch<CW, R>(g0_cplx(s), KRM, jr, sl_cplx(s), sl_cplx(s) + (size_t)KRM * R);
        }
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
                if (p < K) e.y = 0.0;
                e.x -= amax;
                term[p] = a.dc.w[p] * cexp_(e);
            }
        }
        for (int t = warp; t < 2 * np; t += SWARPS) {
            const int s = t >> 1, p = a.bins.ord[p0 + s];
            void* scr = sm + lay.task + (size_t)warp * lay.task_bytes;
            if (s < nr) {
                const double* D = del_real(s) + dj * R * R;
                if (t & 1) z_task<RW, R>(mat_real(s), ldr, jr, D, scr, (RW*)(Zs + s * R * R));
                else ratio_task<RW, R>(mat_real(s), ldr, jr, D, scr, rj, p, CS);
            } else {
                const cxd* D = del_cplx(s) + dj * R * R;
                if (t & 1) z_task<CW, R>(mat_cplx(s), ldr, jr, D, scr, (CW*)(Zs + s * R * R));
                else ratio_task<CW, R>(mat_cplx(s), ldr, jr, D, scr, rj, p, CS);
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
        if (prev) {
            for (int s = 0; s < np; ++s) {
                if (s < nr)
                    pair_update<RW, R>(mat_real(s), ldr, jr, kr, KRM, (const RW*)(Zs + s * R * R),
                                       tables ? sl_real(s) : g0_real(s) + jr, tables ? R : KRM,
                                       tables ? sl_real(s) + (size_t)KRM * R : g0_real(s) + (size_t)jr * KRM,
                                       (RW*)(sm + lay.scratch));
                else
                    pair_update<CW, R>(mat_cplx(s), ldr, jr, kr, KRM, (const CW*)(Zs + s * R * R),
                                       tables ? sl_cplx(s) : g0_cplx(s) + jr, tables ? R : KRM,
                                       tables ? sl_cplx(s) + (size_t)KRM * R : g0_cplx(s) + (size_t)jr * KRM,
                                       (CW*)(sm + lay.scratch));
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
int step_bins(int K, int Kc, int r, int kb, int KRM, size_t rw, size_t cw, size_t smem_max, StepArgs& a, size_t& smem) {
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
            need = step_layout(K + Kc, r, kb, KRM, np, nc, rw, cw, level == 0, level < 2).total;
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
    step_bins(ctx->K, ctx->Kc, ctx->g.r, kmax, kmax * ctx->g.r, fp64 ? 8 : 4, fp64 ? 16 : 8, mx, a, smem);
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
    const int CS = step_bins(ctx->K, ctx->Kc, g.r, kb, a.KRM, fp64 ? 8 : 4, fp64 ? 16 : 8, step_smem_max(ctx), a, smem);
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
