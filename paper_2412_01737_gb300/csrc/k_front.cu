// FP64 log-Pfaffian of M_nm(G) (Sec. 5: N_nm(G) = c_nm Pf(M_nm(G))) by a
// site-by-site elimination that follows the lattice.
//
// M = D + O(G) Gamma_X O(G)^T couples a virtual Majorana only to the other
// Majoranas of its own site (the block D and the link block of its own end)
// and to the partner end of its link.  Sites are added in index order
// s = 0 .. V-1; after adding site s, every Majorana whose site and link
// partner are both added is "closed": no later site couples to it, so it can
// be eliminated from the dense "front" (the Schur complement of M on the
// added, not yet eliminated Majoranas).  With M = [[A, B], [-B^T, C]] and A
// the block of one eliminated pair (k, p),
//     Pf(M) = M_kp Pf(C + (v u^T - u v^T) / M_kp),   u = M[k, rest], v = M[p, rest]
// (Schur complement of a skew matrix), after moving k, p to the front, which
// multiplies Pf by the sign of that permutation.  Pairs are chosen by the
// largest |entry| within a panel of the closed set, as long as that is no
// smaller than 1/16 of what the closed set offers; else the panel ends there
// and the largest entry of the whole remaining closed set comes next (below).
//
// The front of a periodic L x L lattice holds two rows of link ends (the
// +y ends of the last L sites and the -y ends of row 0, which wait for the
// periodic wrap) plus a few ends of the current row: at 16 x 16, n_v = 2 at
// most 152 of the N = 4096 Majoranas, so one matrix costs ~4e7 FP64 FMAs
// instead of the N^3/6 ~ 1.1e10 of a dense Pfaffian.  The front lives in
// shared memory as a packed upper triangle (skew-symmetric storage), one CTA
// per (configuration, pair) item; fronts too large for shared memory use a
// global-memory slice per CTA.
//
// Sign: Pf(M) = sgn(sigma) prod_t M^(t)_{k_t p_t} with sigma the elimination
// sequence (k_1, p_1, k_2, p_2, ...): the sign of the schedule's own sequence
// (known on the host) times one factor -1 per exchange a pivot choice makes.
//
// What bounds it: the FP64 unit (two FMAs per clock and SM).  The closed set (at
// most four links, 32 Majoranas) is
// eliminated in chunks of at most 16 Majoranas: their rows are copied into a
// dense panel over the live slots, the pivoted pairs update the panel only,
// and the rest of the front then takes the chunk's rank-16 update in one
// pass, 2 x 2 register tiles over a list of the live slots.
//
// A chunk of a larger closed set can be nearly singular by itself although the
// closed set is not (the complex pairs n < m; a pivot of 1e-8 then costs eight
// digits).  So a pivot below 1/16 ends such a chunk, its remaining rows go back
// to the front, and the next chunk starts from the largest entry of all that
// is left of the closed set, against which its other pivots are measured.
// Random states of every group have pivots of 0.2 and more there and never
// take that turn.
//
// Against a rank-2
// update of the whole triangle per pair (33 % of the FP64 slots useful: dead
// slots, ragged rows, a shared-memory round trip per product pair) 64 real
// and 96 complex items of 16 x 16, n_v = 2 took 113 ms and take 50,
// 1024 real items of 8 x 8 Z2 10.2 ms and 1.7.  Real and complex items
// run side by side on two streams, because a handful of configurations fills
// only part of the chip with either.  Fronts of at most 48 slots (8 x 8 Z2:
// 44) take 64 threads, so that many items share an SM and the barriers of the
// short steps are cheap; larger ones 256.
#include <algorithm>
#include <vector>
#include "ggf_ctx.h"
#include "ggf_geom.cuh"

namespace {

constexpr int CHUNK = 16;          // closed Majoranas per panel
constexpr int SMALL_FRONT = 48;    // slots up to which an item takes 64 threads
constexpr int MAX_CLOSED = 32;     // Majoranas closed by one site (four links)
enum { SMALL_PIVOT = 1, NO_PIVOT = 2 };
constexpr double PIVOT_FLOOR = 1.0 / 256.0;    // smallest |pivot|^2 of a chunk, over the largest there is

__host__ __device__ __forceinline__ int tri_row(int i, int F) { return i * (2 * F - i - 1) / 2 - i - 1; }

__device__ __forceinline__ double fsq(double v) { return v * v; }
__device__ __forceinline__ double fsq(cxd v) { return fma(v.x, v.x, v.y * v.y); }
__device__ __forceinline__ double fneg(double v) { return -v; }
__device__ __forceinline__ cxd fneg(cxd v) { return {-v.x, -v.y}; }
__device__ __forceinline__ double finv(double v) { return 1.0 / v; }
__device__ __forceinline__ cxd finv(cxd v) { return cxd{1.0, 0.0} / v; }
__device__ __forceinline__ double fmul(double a, double b) { return a * b; }
__device__ __forceinline__ cxd fmul(cxd a, cxd b) { return a * b; }
__device__ __forceinline__ cxd as_c(double v) { return {v, 0.0}; }
__device__ __forceinline__ cxd as_c(cxd v) { return v; }
// r += a * b - c * d
__device__ __forceinline__ void frank2(double& r, double a, double b, double c, double d) {
    r = fma(a, b, r);
    r = fma(-c, d, r);
}
__device__ __forceinline__ void frank2(cxd& r, cxd a, cxd b, cxd c, cxd d) {
    double x = r.x, y = r.y;
    x = fma(a.x, b.x, x); x = fma(-a.y, b.y, x); x = fma(-c.x, d.x, x); x = fma(c.y, d.y, x);
    y = fma(a.x, b.y, y); y = fma(a.y, b.x, y); y = fma(-c.x, d.y, y); y = fma(-c.y, d.x, y);
    r = {x, y};
}

// S(a, b) of the packed strict upper triangle, skew-symmetric
template <class T>
__device__ __forceinline__ T sget(const T* S, int F, int a, int b) {
    if (a < b) return S[tri_row(a, F) + b];
    if (a > b) return fneg(S[tri_row(b, F) + a]);
    return Sc<T>::zero();
}

// Largest |get(x, y)|^2 over x < y < n (n <= 32, one warp): best in every lane,
// at = 32 x + y.  NaN orders above all others.
template <class Get>
__device__ __forceinline__ void warp_best_pair(int n, Get get, double& best, int& at) {
    best = -1.0;
    at = 1;
    for (int p = threadIdx.x & 31; p < n * (n - 1) / 2; p += 32) {
        int y = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)p)) * 0.5f);
        if (y * (y - 1) / 2 > p) --y;
        if ((y + 1) * y / 2 <= p) ++y;
        const int x = p - y * (y - 1) / 2;
        const double m = fsq(get(x, y));
        if (m > best || !(m == m)) { best = m; at = x * 32 + y; }
    }
    const unsigned key = best >= 0.0 || !(best == best) ? (unsigned)__double2hiint(best) & 0x7fffffffu : 0u;
    const unsigned top = __reduce_max_sync(0xffffffffu, key);
    const int src = __ffs(__ballot_sync(0xffffffffu, key == top && !(best < 0.0))) - 1;
    best = __shfl_sync(0xffffffffu, best, src);
    at = __shfl_sync(0xffffffffu, at, src);
}

// The pair (x, y), x < y, of list a, values (k, p), to its first two positions;
// whether that is an odd permutation.
__device__ __forceinline__ bool pair_to_front(int* a, int x, int y, int& k, int& p) {
    k = a[x];
    p = a[y];
    a[x] = a[0];
    a[0] = k;
    a[y] = a[1];
    a[1] = p;
    return (x > 0) != (y > 1);
}

struct FrontArgs {
    int F;              // slots of the front
    int N, B, V;
    const int* slot;    // [N] slot of Majorana i (fixed by the schedule)
    const int* eoff;    // [V + 1] offsets into elim
    const int* elim;    // slots eliminated after adding site s
    int sign;           // of the schedule's elimination sequence
};

// The four link ends of the site being added: link, its value's twist.
struct EndTab {
    int link;
    double gval;
    double tw[16];      // U(1): cos, sin of q_j theta; SU(2): doublet rotation
};

// M(i, j) for Majorana a of site s (i = s B + a) and any Majorana j.
template <class T>
__device__ __forceinline__ T front_entry(const DevConst& dc, int pair, const EndTab* tab, int s, int a, int j) {
    const Geometry& g = dc.g;
    const int e = a / g.h2, x = a - e * g.h2;
    const int l = tab[e].link, pi = (e & 1) ? x : g.h2 + x;
    T v = Sc<T>::zero();
    int lj, pj;
    if (j / g.B == s) {
        const int b = j - s * g.B, eb = b / g.h2, xb = b - eb * g.h2;
        v = Sc<T>::from(Sc<double>::to(dc.D[((size_t)s * g.B + a) * g.B + b]));
        lj = tab[eb].link;
        pj = (eb & 1) ? xb : g.h2 + xb;
    } else {
        link_of(g, j, lj, pj);
    }
    if (lj == l)
        v += g.group == GGF_SU2 ? twisted_su2<T>(dc, pair, l, pi, pj, tab[e].tw)
                                : twisted_tab<T>(dc, pair, l, pi, pj, tab[e].gval, tab[e].tw);
    return v;
}

// Byte offsets of an item's shared arrays.
struct FrontLayout {
    size_t tab, idx, lv, tri, total;
};
__host__ __device__ inline FrontLayout front_layout(int F, size_t elem, bool tri) {
    FrontLayout l;
    size_t o = (size_t)CHUNK * F * elem;       // the panel comes first
    auto take = [&](size_t& at, size_t bytes) { at = o; o = (o + bytes + 15) & ~(size_t)15; };
    take(l.tab, 4 * sizeof(EndTab));
    take(l.idx, (size_t)F * sizeof(int));
    take(l.lv, (size_t)F * sizeof(unsigned short));
    take(l.tri, tri ? (size_t)F * (F - 1) / 2 * elem : 0);
    l.total = o;
    return l;
}

// One CTA per item (grid-stride); item = q npf + pair of configuration
// chains[q] (or q).  Its log-weight goes to ell[q][pair_off + pair]; items
// without a usable pivot are appended to bad[1 ..], counted in bad[0].
// WIDE: some site closes more than CHUNK Majoranas (n_v = 2); without it every
// chunk is a whole closed set.
template <class T, int NT, bool WIDE>
__global__ void __launch_bounds__(NT, NT == 64 ? 8 : (sizeof(T) == 8 ? 2 : 1))
front_pf_kernel(DevConst dc, FrontArgs fa, long long n_items, const int* chains, int npf, int pair_off,
                const void* links, cxd* ell, int* bad, T* gws, size_t tri_elems, int in_smem) {
    extern __shared__ __align__(16) unsigned char fsm[];
    __shared__ int s_end, s_done, s_nl;        // s_end: how the chunk ended, s_done: after how many rows
    __shared__ T s_inv;
    __shared__ T s_scale[CHUNK];
    __shared__ int ord[CHUNK], es[CHUNK], cl[MAX_CLOSED];
    constexpr int NW = NT / 32;
    const int F = fa.F, B = fa.B, V = fa.V;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const FrontLayout lay = front_layout(F, sizeof(T), in_smem != 0);
    T* Pn = (T*)fsm;                                     // [CHUNK][F]
    EndTab* tab = (EndTab*)(fsm + lay.tab);
    int* idx = (int*)(fsm + lay.idx);                    // Majorana of a slot, -1: dead
    unsigned short* lv = (unsigned short*)(fsm + lay.lv);
    T* S = in_smem ? (T*)(fsm + lay.tri) : gws + (size_t)blockIdx.x * tri_elems;
    const Geometry& g = dc.g;
    for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int q = (int)(item / npf), pair = (int)(item - (long long)q * npf);
        const int cfg = chains ? chains[q] : q;
        for (int a = tid; a < F; a += NT) idx[a] = -1;
        if (tid == 0) s_end = 0;
        __syncthreads();
        // lane 0 of warp 0: prod of the pivots as pr 2^ex
        cxd pr = {(double)fa.sign, 0.0};
        long long ex = 0;
        for (int s = 0; s < V; ++s) {
            // ---- add site s: its B Majoranas take their slots, their rows are M's entries
            if (tid < 4) {
                EndTab& t = tab[tid];
                int pos;
                link_of(g, s * B + tid * g.h2, t.link, pos);
                t.gval = 1.0;
                if (g.group == GGF_Z2) {
                    t.gval = (double)((const int8_t*)links)[(size_t)cfg * g.n_links + t.link];
                } else if (g.group == GGF_U1) {
                    const double th = ((const double*)links)[(size_t)cfg * g.n_links + t.link];
                    for (int j = 0; j < g.n_v; ++j) sincos(g.q[j] * th, &t.tw[2 * j + 1], &t.tw[2 * j]);
                } else {
                    doublet_rotation(link_quat(g, links, cfg, t.link), t.tw);
                }
            }
            for (int k = tid; k < B; k += NT) idx[fa.slot[s * B + k]] = s * B + k;
            const int first = fa.eoff[s], ne = fa.eoff[s + 1] - first;
            if (WIDE && ne > CHUNK)
                for (int k = tid; k < ne; k += NT) cl[k] = fa.elim[first + k];
            __syncthreads();
            for (int k = warp; k < B; k += NW) {
                const int a = fa.slot[s * B + k];
                for (int b = lane; b < F; b += 32) {
                    const int jb = idx[b];
                    if (b == a || jb < 0) continue;
                    if (jb >= s * B && b < a) continue;        // new-new pair: written once, by the lower slot's row
                    const T val = front_entry<T>(dc, pair, tab, s, k, jb);
                    if (a < b) S[tri_row(a, F) + b] = val;
                    else S[tri_row(b, F) + a] = fneg(val);
                }
            }
            __syncthreads();
            // ---- eliminate the closed Majoranas, a chunk at a time
            int e = 0;
            bool search = false;       // the last chunk ended at a small pivot
            while (e < ne) {
                const int c = min(CHUNK, ne - e);
                // (warp 0) |pivot|^2 below which this chunk ends: its upper word, which
                // orders as an integer and leaves the FP64 unit alone
                int low = __double2hiint(PIVOT_FLOOR);
                if (WIDE && search) {
                    if (warp == 0) {
                        double best;
                        int bq;
                        warp_best_pair(ne - e, [&](int x, int y) { return sget(S, F, cl[e + x], cl[e + y]); }, best, bq);
                        low = __double2hiint(PIVOT_FLOOR * best);
                        int k, p;
                        if (lane == 0 && pair_to_front(cl + e, bq / 32, bq % 32, k, p)) pr = -pr;
                    }
                    __syncthreads();
                }
                if (WIDE && tid == 0) s_end = 0;
                if (tid < c) { es[tid] = WIDE && ne > CHUNK ? cl[e + tid] : fa.elim[first + e + tid]; ord[tid] = tid; }
                __syncthreads();
                if (tid < c) idx[es[tid]] = -1;
                __syncthreads();
                if (warp == 0) {                        // the live slots, ascending
                    int n = 0;
                    for (int b0 = 0; b0 < F; b0 += 32) {
                        const bool live = b0 + lane < F && idx[b0 + lane] >= 0;
                        const unsigned m = __ballot_sync(0xffffffffu, live);
                        if (live) lv[n + __popc(m & ((1u << lane) - 1u))] = (unsigned short)(b0 + lane);
                        n += __popc(m);
                    }
                    if (lane == 0) s_nl = n;
                }
                __syncthreads();
                const int nl = s_nl, W = c + nl;
                for (int t = warp; t < c; t += NW)
                    for (int w = lane; w < W; w += 32)
                        Pn[(size_t)t * F + w] = sget(S, F, es[t], w < c ? es[w] : lv[w - c]);
                __syncthreads();
                for (int t = 0; t < c; t += 2) {
                    if (warp == 0) {
                        // pivot: the largest entry among the chunk's remaining pairs
                        double best;
                        int bq;
                        warp_best_pair(c - t, [&](int x, int y) { return Pn[(size_t)ord[t + x] * F + ord[t + y]]; }, best, bq);
                        if (WIDE && e + c < ne && __double2hiint(best) < low && !(search && t == 0)) {
                            if (lane == 0) { s_end = SMALL_PIVOT; s_done = t; }     // better ones may lie outside the chunk
                        } else if (lane == 0) {
                            if (!(best > 1e-16) || !isfinite(best)) s_end = NO_PIVOT;   // no usable pivot: refactor densely
                            int k, p;
                            const bool odd = pair_to_front(ord + t, bq / 32, bq % 32, k, p);
                            const T akp = Pn[(size_t)k * F + p];
                            const T inv = finv(akp);
                            s_inv = inv;
                            s_scale[t] = inv;
                            pr = pr * as_c(akp);
                            if (odd) pr = -pr;
                            // keep the product in range by its own power of two
                            const int ep = ((__double2hiint(fmax(fabs(pr.x), fabs(pr.y))) >> 20) & 0x7ff) - 1023;
                            const double sc = __hiloint2double((1023 - ep) << 20, 0);
                            pr = {pr.x * sc, pr.y * sc};
                            ex += ep;
                        }
                    }
                    __syncthreads();
                    if (s_end) break;
                    // the remaining rows of the chunk: R += (v_R / a) k - (k_R / a) v
                    const T* rk = Pn + (size_t)ord[t] * F;
                    const T* rp = Pn + (size_t)ord[t + 1] * F;
                    const T inv = s_inv;
                    for (int i = t + 2 + warp; i < c; i += NW) {
                        const int row = ord[i];
                        const T vi = fmul(rp[row], inv), ki = fmul(rk[row], inv);
                        T* r = Pn + (size_t)row * F;
                        for (int w = lane; w < W; w += 32) {
                            T x = r[w];
                            frank2(x, vi, rk[w], ki, rp[w]);
                            r[w] = x;
                        }
                    }
                    __syncthreads();
                }
                if (s_end == NO_PIVOT) break;
                int done = c;
                if (WIDE && s_end == SMALL_PIVOT) {
                    // the rows that the chunk leaves behind: back to the front, and zero in
                    // the panel, so that the update below takes nothing from them
                    done = s_done;
                    for (int i = done + warp; i < c; i += NW) {
                        const int row = ord[i], a = es[row];
                        for (int w = i + 1 + lane; w < W; w += 32) {
                            const int col = w < c ? ord[w] : w, b = w < c ? es[col] : lv[w - c];
                            const T val = Pn[(size_t)row * F + col];
                            if (a < b) S[tri_row(a, F) + b] = val;
                            else S[tri_row(b, F) + a] = fneg(val);
                            if (w >= c) Pn[(size_t)row * F + col] = Sc<T>::zero();
                        }
                        if (lane == 0) {
                            s_scale[i] = Sc<T>::zero();
                            cl[e + i] = a;
                            idx[a] = 0;        // live again (which Majorana it is matters only to later sites)
                        }
                    }
                    __syncthreads();
                }
                // u_t = row k_t / a_t over the live columns
                for (int t = 2 * warp; t < c; t += 2 * NW) {
                    T* r = Pn + (size_t)ord[t] * F + c;
                    const T inv = s_scale[t];
                    for (int w = lane; w < nl; w += 32) r[w] = fmul(r[w], inv);
                }
                __syncthreads();
                // C += sum_t v_t u_t^T - u_t v_t^T on the pairs of live slots (nl is
                // even: link ends hold 2 n_v Majoranas), 2 x 2 per thread and turn
                const int th = nl >> 1;
                for (int id = tid; id < th * (th + 1) / 2; id += NT) {
                    int tj = (int)((sqrtf(8.0f * (float)id + 1.0f) - 1.0f) * 0.5f);
                    if (tj * (tj + 1) / 2 > id) --tj;
                    if ((tj + 1) * (tj + 2) / 2 <= id) ++tj;
                    const int i = 2 * (id - tj * (tj + 1) / 2), j = 2 * tj;
                    const int r0 = lv[i], r1 = lv[i + 1], c0 = lv[j], c1 = lv[j + 1];
                    T* S0 = S + tri_row(r0, F);
                    T* S1 = S + tri_row(r1, F);
                    const bool diag = i == j;
                    T a00 = diag ? Sc<T>::zero() : S0[c0], a01 = S0[c1];
                    T a10 = diag ? Sc<T>::zero() : S1[c0], a11 = diag ? Sc<T>::zero() : S1[c1];
                    for (int t = 0; t < c; t += 2) {
                        const T* u = Pn + (size_t)ord[t] * F + c;
                        const T* v = Pn + (size_t)ord[t + 1] * F + c;
                        const T ui0 = u[i], ui1 = u[i + 1], vi0 = v[i], vi1 = v[i + 1];
                        const T uj0 = u[j], uj1 = u[j + 1], vj0 = v[j], vj1 = v[j + 1];
                        frank2(a00, vi0, uj0, ui0, vj0);
                        frank2(a01, vi0, uj1, ui0, vj1);
                        frank2(a10, vi1, uj0, ui1, vj0);
                        frank2(a11, vi1, uj1, ui1, vj1);
                    }
                    S0[c1] = a01;
                    if (!diag) { S0[c0] = a00; S1[c0] = a10; S1[c1] = a11; }
                }
                __syncthreads();
                search = done < c;
                e += done;
            }
            if (s_end == NO_PIVOT) break;
        }
        if (tid == 0) {
            cxd* dst = ell + (size_t)q * dc.P + pair_off + pair;
            if (s_end == NO_PIVOT) {
                *dst = {NAN, 0.0};
                bad[1 + atomicAdd(bad, 1)] = (int)((long long)q * dc.P + pair_off + pair);
            } else {
                const double m = Sc<T>::CPLX ? hypot(pr.x, pr.y) : fabs(pr.x);
                *dst = {log(m) + (double)ex * 0.69314718055994530942, Sc<T>::CPLX ? atan2(pr.y, pr.x) : 0.0};
            }
        }
        __syncthreads();
    }
}

// Elimination schedule for an L x L lattice with B virtual Majoranas per
// site: slot of every Majorana, the slots closed after each site (both ends of
// a link together, so that a chunk holds whole links) and the sign of the
// sequence.
void build_schedule(const Geometry& g, int& F, std::vector<int>& slot, std::vector<int>& eoff, std::vector<int>& elim,
                    int& sign) {
    const int B = g.B, V = g.V, N = g.N, L = g.L;
    slot.assign(N, -1);
    eoff.assign(V + 1, 0);
    elim.clear();
    auto partner_site = [&](int s, int e) {
        const int x = s % L, y = s / L, d = e >> 1;
        if (e & 1) return d == 0 ? y * L + (x + 1) % L : ((y + 1) % L) * L + x;
        return d == 0 ? y * L + (x + L - 1) % L : ((y + L - 1) % L) * L + x;
    };
    auto link_id = [&](int i) {
        const int s = i / B, e = (i % B) / g.h2, d = e >> 1;
        return 2 * ((e & 1) ? s : partner_site(s, e)) + d;
    };
    std::vector<int> free_slots, front, seq;
    int next = 0;
    F = 0;
    for (int s = 0; s < V; ++s) {
        for (int k = 0; k < B; ++k) {
            int sl;
            if (!free_slots.empty()) {
                auto it = std::min_element(free_slots.begin(), free_slots.end());
                sl = *it;
                free_slots.erase(it);
            } else {
                sl = next++;
            }
            slot[s * B + k] = sl;
            front.push_back(s * B + k);
        }
        F = std::max(F, next);
        std::vector<int> keep, closed;
        for (int i : front) {
            const int si = i / B, e = (i % B) / g.h2;
            if (partner_site(si, e) <= s) closed.push_back(i);
            else keep.push_back(i);
        }
        std::stable_sort(closed.begin(), closed.end(), [&](int a, int b) { return link_id(a) < link_id(b); });
        for (int i : closed) {
            elim.push_back(slot[i]);
            free_slots.push_back(slot[i]);
            seq.push_back(i);
        }
        front.swap(keep);
        eoff[s + 1] = (int)elim.size();
    }
    // sign of the permutation by its cycles
    std::vector<char> seen(seq.size(), 0);
    int cycles = 0;
    for (size_t i = 0; i < seq.size(); ++i) {
        if (seen[i]) continue;
        ++cycles;
        for (size_t j = i; !seen[j]; j = (size_t)seq[j]) seen[j] = 1;
    }
    sign = ((int)seq.size() - cycles) % 2 ? -1 : 1;
}

// opt-in shared memory per CTA (227 KB) less a margin for the static variables
const size_t kSmemMax = 227 * 1024 - 1024;

template <class T, int NT>
ggf_status raise_cap(ggf_ctx* ctx) {
    GGF_CK(cudaFuncSetAttribute(front_pf_kernel<T, NT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
    GGF_CK(cudaFuncSetAttribute(front_pf_kernel<T, NT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
    return GGF_OK;
}

}  // namespace

ggf_status ggf_front_prepare(ggf_ctx* ctx) {
    const Geometry& g = ctx->g;
    if (ctx->d_front && ctx->front_L == g.L && ctx->front_B == g.B) return GGF_OK;
    if (ctx->d_front) cudaFree(ctx->d_front);
    ctx->d_front = nullptr;
    int F = 0, sign = 1;
    std::vector<int> slot, eoff, elim;
    build_schedule(g, F, slot, eoff, elim, sign);
    if ((int)elim.size() != g.N) return ggf_fail(ctx, GGF_ESTATE, "front schedule does not close every Majorana");
    int closed = 0;
    for (int s = 0; s < g.V; ++s) closed = std::max(closed, eoff[s + 1] - eoff[s]);
    if (closed > MAX_CLOSED) return ggf_fail(ctx, GGF_ESTATE, "front schedule closes too many Majoranas");
    std::vector<int> all;
    all.insert(all.end(), slot.begin(), slot.end());
    all.insert(all.end(), eoff.begin(), eoff.end());
    all.insert(all.end(), elim.begin(), elim.end());
    GGF_CK(cudaMalloc(&ctx->d_front, all.size() * sizeof(int)));
    GGF_CK(cudaMemcpy(ctx->d_front, all.data(), all.size() * sizeof(int), cudaMemcpyHostToDevice));
    if (!ctx->front_st) {
        GGF_CK(cudaStreamCreateWithFlags(&ctx->front_st, cudaStreamNonBlocking));
        GGF_CK(cudaEventCreateWithFlags(&ctx->front_fork, cudaEventDisableTiming));
        GGF_CK(cudaEventCreateWithFlags(&ctx->front_join, cudaEventDisableTiming));
    }
    ctx->front_F = F;
    ctx->front_wide = closed > CHUNK;
    ctx->front_sign = sign;
    ctx->front_L = g.L;
    ctx->front_B = g.B;
    static bool attr_done[64] = {false};
    if (ctx->device >= 0 && ctx->device < 64 && !attr_done[ctx->device]) {
        GGF_TRY((raise_cap<double, 64>(ctx)));
        GGF_TRY((raise_cap<double, 256>(ctx)));
        GGF_TRY((raise_cap<cxd, 64>(ctx)));
        GGF_TRY((raise_cap<cxd, 256>(ctx)));
        attr_done[ctx->device] = true;
    }
    return GGF_OK;
}

void ggf_front_free(ggf_ctx* ctx) {
    if (ctx->d_front) cudaFree(ctx->d_front);
    if (ctx->front_ws) cudaFree(ctx->front_ws);
    if (ctx->front_st) cudaStreamDestroy(ctx->front_st);
    if (ctx->front_fork) cudaEventDestroy(ctx->front_fork);
    if (ctx->front_join) cudaEventDestroy(ctx->front_join);
    ctx->d_front = nullptr;
    ctx->front_ws = nullptr;
    ctx->front_ws_bytes = 0;
    ctx->front_st = nullptr;
    ctx->front_fork = ctx->front_join = nullptr;
    ctx->front_L = ctx->front_B = -1;
}

// log Pf(M_nm(G)) of every pair of n configurations (d_chains[q], or q where
// d_chains is null) of d_links into d_ell [n][P]: (log|Pf|, phase).  Items
// whose closed sets had no usable pivot are listed in d_bad (1 + n P ints:
// the count, then positions in d_ell; the caller refactors those densely).
ggf_status ggf_front_pfaffian(ggf_ctx* ctx, int n, const int* d_chains, const void* d_links, cxd* d_ell, int* d_bad,
                              cudaStream_t st) {
    if (n == 0) return GGF_OK;
    GGF_TRY(ggf_front_prepare(ctx));
    const Geometry& g = ctx->g;
    const int F = ctx->front_F, sms = ctx->n_sms > 0 ? ctx->n_sms : 152;
    FrontArgs fa;
    fa.F = F;
    fa.N = g.N;
    fa.B = g.B;
    fa.V = g.V;
    fa.slot = ctx->d_front;
    fa.eoff = ctx->d_front + g.N;
    fa.elim = ctx->d_front + g.N + g.V + 1;
    fa.sign = ctx->front_sign;
    const size_t tri = (size_t)F * (F - 1) / 2;
    int grid[2];
    bool in_smem[2];
    size_t need = 0, off[2] = {0, 0};
    for (int f = 0; f < 2; ++f) {
        const size_t elem = f ? sizeof(cxd) : sizeof(double);
        const long long items = (long long)n * (f ? ctx->Kc : ctx->K);
        in_smem[f] = front_layout(F, elem, true).total <= kSmemMax;
        grid[f] = (int)std::min<long long>(items, in_smem[f] ? 1 << 20 : 2 * sms);
        off[f] = need;
        if (!in_smem[f]) need += ((size_t)grid[f] * tri * elem + 255) / 256 * 256;
    }
    if (need > ctx->front_ws_bytes) {
        if (ctx->front_ws) cudaFree(ctx->front_ws);
        ctx->front_ws = nullptr;
        ctx->front_ws_bytes = 0;
        GGF_CK(cudaMalloc(&ctx->front_ws, need));
        ctx->front_ws_bytes = need;
    }
    GGF_CK(cudaMemsetAsync(d_bad, 0, sizeof(int), st));
    const bool both = ctx->Kc > 0;
    if (both) {
        GGF_CK(cudaEventRecord(ctx->front_fork, st));
        GGF_CK(cudaStreamWaitEvent(ctx->front_st, ctx->front_fork, 0));
    }
    const bool small = F <= SMALL_FRONT;
#define GGF_FRONT(T, NT, W, f, npf, off_p, stream)                                                               \
    front_pf_kernel<T, NT, W><<<grid[f], NT, front_layout(F, sizeof(T), in_smem[f]).total, stream>>>(                \
        ctx->dc(), fa, (long long)n * (npf), d_chains, npf, off_p, d_links, d_ell, d_bad,                         \
        (T*)((unsigned char*)ctx->front_ws + off[f]), tri, in_smem[f] ? 1 : 0)
#define GGF_FRONTS(T, f, npf, off_p, stream)                                                                      \
    do {                                                                                                          \
        if (ctx->front_wide) {                                                                                    \
            if (small) GGF_FRONT(T, 64, true, f, npf, off_p, stream);                                             \
            else GGF_FRONT(T, 256, true, f, npf, off_p, stream);                                                  \
        } else {                                                                                                  \
            if (small) GGF_FRONT(T, 64, false, f, npf, off_p, stream);                                            \
            else GGF_FRONT(T, 256, false, f, npf, off_p, stream);                                                 \
        }                                                                                                         \
    } while (0)
    if (both) {      // the complex items, four times as long, are placed first
        GGF_FRONTS(cxd, 1, ctx->Kc, ctx->K, st);
        GGF_CK(cudaGetLastError());
    }
    cudaStream_t rs = both ? ctx->front_st : st;
    GGF_FRONTS(double, 0, ctx->K, 0, rs);
    GGF_CK(cudaGetLastError());
#undef GGF_FRONTS
#undef GGF_FRONT
    ctx->launches += both ? 2 : 1;
    if (both) {
        GGF_CK(cudaEventRecord(ctx->front_join, ctx->front_st));
        GGF_CK(cudaStreamWaitEvent(st, ctx->front_join, 0));
    }
    return GGF_OK;
}
