// FP64 inverses W = M_nm(G)^{-1} along the lattice (start and refresh of FP64
// chains).
//
// Without its y links, M falls into L blocks of one lattice row each (size
// b = L B).  Those are inverted densely (b^3 each), and neighbouring groups of
// rows are then joined, pairwise, by adding the y links between them: a change
// Delta of M on the ends T = T_0 u T_1 of those links (kT = L h2 Majoranas per
// group and boundary, two boundaries where the last joint closes the torus),
//     W' = W - W[:, T] Z W[T, :],   Z = (1 + Delta W_TT)^{-1} Delta,
// with W block diagonal before, so that block (g, g') of the change has rank
// kT:  - W_g[:, T_g] Z_gg' W_g'[T_g', :].  The joints cost N^2 (kT + kT / 4 + ...)
// FMAs instead of the N^3 of Gauss-Jordan (N = 4096: 26 times fewer), and half
// of that again because W is antisymmetric: only tiles on and above the
// diagonal are formed, the others are their negative transposes.
//
// Accuracy: the open row blocks can be worse conditioned than M (residuals of
// 1e-16 .. 1e-11 over random symmetric states, against 1e-15 of a pivoted
// elimination), so the result is refined: R = I - M W in FP64 from the sparse
// M, W <- W + W R with the product on the tensor cores from FP32 copies (the
// three-product split, 1e-6 relative: a residual r becomes about 1e-6 r plus
// the FP64 floor of R).  Matrices whose residual stays above 1e-12 go to
// the dense Gauss-Jordan elimination.
//
// What bounds it: the FP64 unit in the joints, kernel launches for small
// batches.  Measured, 8 configurations of 8 x 8 U(1), n_v = 2, K = 2 (16 real
// and 8 complex matrices of order 1024): 190 ms by Gauss-Jordan, 22 ms so;
// the start of one chain of 16 x 16 U(1), K = 4 (4 real and 6 complex ones of
// order 4096): 6.0 s and 0.30 s.
#include <algorithm>
#include <vector>
#include "ggf_ctx.h"
#include "ggf_geom.cuh"

size_t ggf_factor_tmp_bytes(int n, int batch);
size_t ggf_flush_ps_item_bytes(ggf_ctx* ctx, bool cplx);
ggf_status ggf_flush_tc_items(ggf_ctx* ctx, bool cplx, int n, float* W, const int* wmap, const float* Pan,
                              const int* pend, int terms, unsigned char* ps, cudaStream_t st);

namespace {

// One joint: rows y0 .. ym - 1 and ym .. y1 - 1; cyc: also across the torus.
struct Joint {
    int y0, ym, y1, cyc;
};

__device__ __forceinline__ void mac(double& r, double a, double b) { r = fma(a, b, r); }
__device__ __forceinline__ void mac(cxd& r, cxd a, cxd b) {
    r.x = fma(a.x, b.x, r.x); r.x = fma(-a.y, b.y, r.x);
    r.y = fma(a.x, b.y, r.y); r.y = fma(a.y, b.x, r.y);
}

// Majorana t of T_g: boundary t / LH (0: between ym - 1 and ym, 1: the torus),
// column x of the lattice, mode k of the end.  src: whether it is a source end.
__device__ __forceinline__ int joint_majorana(const Geometry& g, const Joint& jt, int grp, int t, int& link, int& pos) {
    const int LH = g.L * g.h2, bd = t / LH, x = (t - bd * LH) / g.h2, k = t % g.h2;
    const int src_row = bd ? jt.y1 - 1 : jt.ym - 1, dst_row = bd ? jt.y0 : jt.ym;
    const bool src = (grp == 0) == (bd == 0);
    link = bd * g.L + x;
    pos = src ? k : g.h2 + k;
    return ((src ? src_row : dst_row) * g.L + x) * g.B + (src ? 3 : 2) * g.h2 + k;
}

// Row blocks without the y links: Rb[item L + y][b][b].
template <class T>
__global__ void row_blocks(DevConst dc, const int* cfg, const int* pair, const void* links, T* Rb) {
    const Geometry& g = dc.g;
    const int b = g.L * g.B, it = blockIdx.y / g.L, y = blockIdx.y % g.L;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= b * b) return;
    const int i = y * b + e / b, j = y * b + e % b;
    T v = Sc<T>::zero();
    const int si = i / g.B, sj = j / g.B;
    int li, pi, lj, pj;
    link_of(g, i, li, pi);
    link_of(g, j, lj, pj);
    if (si == sj || (li == lj && (li & 1) == 0)) {
        if (li == lj && (li & 1)) v = Sc<T>::from(Sc<double>::to(dc.D[((size_t)si * g.B + i % g.B) * g.B + j % g.B]));
        else v = assemble_elem<T>(dc, links, cfg[it], pair[it], i, j);
    }
    Rb[(size_t)blockIdx.y * b * b + e] = v;
}

template <class T>
__global__ void place_rows(int N, int b, int L, const T* Rb, T* A) {
    const int it = blockIdx.y / L, y = blockIdx.y % L;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= b * b) return;
    A[(size_t)it * N * N + (size_t)(y * b + e / b) * N + y * b + e % b] = Rb[(size_t)blockIdx.y * b * b + e];
}

// Delta blocks of a level's links: D[(joint, item)][link][r][r].
template <class T>
__global__ void joint_delta(DevConst dc, const Joint* joints, int items, const int* cfg, const int* pair,
                            const void* links, int nlk, T* D) {
    const Geometry& g = dc.g;
    const int mi = blockIdx.y, it = mi % items, r = g.r;
    const Joint jt = joints[mi / items];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nlk * r * r) return;
    const int k = e / (r * r), x = k % g.L, bd = k / g.L;
    const int l = 2 * ((bd ? jt.y1 - 1 : jt.ym - 1) * g.L + x) + 1, xi = e / r % r, yi = e % r;
    T v;
    if (g.group == GGF_SU2) {
        double R[16];
        doublet_rotation(link_quat(g, links, cfg[it], l), R);
        v = twisted_su2<T>(dc, pair[it], l, xi, yi, R);
    } else {
        double gv, th;
        link_value<T>(dc, links, cfg[it], l, gv, th);
        v = twisted<T>(dc, pair[it], l, xi, yi, gv, th);
    }
    D[(size_t)mi * nlk * r * r + e] = v;
}

// S = 1 + Delta W_TT (2 kT x 2 kT) of every (joint, item).
template <class T>
__global__ void joint_small(Geometry g, const Joint* joints, int items, int kT, int nlk, const T* A, const T* D, T* S) {
    const int mi = blockIdx.y, N = g.N, r = g.r, k2 = 2 * kT;
    const Joint jt = joints[mi / items];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= k2 * k2) return;
    const int a = e / k2, c = e % k2, ga = a / kT, gc = c / kT;
    int la, pa, lc, pc;
    joint_majorana(g, jt, ga, a % kT, la, pa);
    const int jc = joint_majorana(g, jt, gc, c % kT, lc, pc);
    const T* W = A + (size_t)(mi % items) * N * N;
    const T* Db = D + ((size_t)mi * nlk + la) * r * r + pa * r;
    T v = a == c ? Sc<T>::one() : Sc<T>::zero();
    // the link's Majoranas in group gc: W couples T within a group only
    const int t0 = (la / g.L) * g.L * g.h2 + (la % g.L) * g.h2;
    for (int k = 0; k < g.h2; ++k) {
        int lk, pk;
        const int i = joint_majorana(g, jt, gc, t0 + k, lk, pk);
        mac(v, Db[pk], W[(size_t)i * N + jc]);
    }
    S[(size_t)mi * k2 * k2 + e] = v;
}

// Z = S^{-1} Delta.
template <class T>
__global__ void joint_z(Geometry g, const Joint* joints, int items, int kT, int nlk, const T* Si, const T* D, T* Z) {
    const int mi = blockIdx.y, r = g.r, k2 = 2 * kT;
    const Joint jt = joints[mi / items];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= k2 * k2) return;
    const int a = e / k2, c = e % k2;
    int lc, pc;
    joint_majorana(g, jt, c / kT, c % kT, lc, pc);
    const T* Db = D + ((size_t)mi * nlk + lc) * r * r + pc;
    const T* Sr = Si + (size_t)mi * k2 * k2 + (size_t)a * k2;
    const int t0 = (lc / g.L) * g.L * g.h2 + (lc % g.L) * g.h2;
    T v = Sc<T>::zero();
    for (int gg = 0; gg < 2; ++gg)
        for (int k = 0; k < g.h2; ++k) {
            int lk, pk;
            joint_majorana(g, jt, gg, t0 + k, lk, pk);
            mac(v, Sr[gg * kT + t0 + k], Db[(size_t)pk * r]);
        }
    Z[(size_t)mi * k2 * k2 + e] = v;
}

// P[(joint, item)][i][t] = W[i][T_g(i) t], rows i of the joint (i from y0 b).
template <class T>
__global__ void joint_cols(Geometry g, const Joint* joints, int items, int kT, const T* A, T* P) {
    const int mi = blockIdx.y, N = g.N, b = g.L * g.B;
    const Joint jt = joints[mi / items];
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(e / kT), t = (int)(e % kT), n = (jt.y1 - jt.y0) * b;
    if (i >= n) return;
    int l, p;
    const int j = joint_majorana(g, jt, i >= (jt.ym - jt.y0) * b, t, l, p);
    P[((size_t)(mi % items) * N + jt.y0 * b + i) * kT + t] = A[(size_t)(mi % items) * N * N + (size_t)(jt.y0 * b + i) * N + j];
}

// 64 x 64 tile products, 256 threads as 16 x 16 with 4 x 4 results each (rows
// ty + 16 u, columns tx + 16 v: neighbouring threads read neighbouring words).
constexpr int GT = 64, GK = 16;

template <class T, class LA, class LB>
__device__ __forceinline__ void tile_product(int K, T (&acc)[4][4], T (*As)[GT + 1], T (*Bs)[GT + 1], LA la, LB lb) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = Sc<T>::zero();
    for (int k0 = 0; k0 < K; k0 += GK) {
        for (int e = threadIdx.x; e < GK * GT; e += 256) {
            const int ka = e % GK, ra = e / GK;          // A: row-major, rank contiguous
            As[ka][ra] = k0 + ka < K ? la(ra, k0 + ka) : Sc<T>::zero();
            const int kb = e / GT, cb = e % GT;          // B: rank-major, columns contiguous
            Bs[kb][cb] = k0 + kb < K ? lb(k0 + kb, cb) : Sc<T>::zero();
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < GK; ++k) {
            T av[4], bv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) av[u] = As[k][ty + 16 * u];
#pragma unroll
            for (int v = 0; v < 4; ++v) bv[v] = Bs[k][tx + 16 * v];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) mac(acc[u][v], av[u], bv[v]);
        }
        __syncthreads();
    }
}

// Tile q of a joint's rows: tiles never straddle the two groups.
__device__ __forceinline__ bool joint_tile(int n1, int n2, int q, int& i0, int& n, int& grp) {
    const int q1 = (n1 + GT - 1) / GT, q2 = (n2 + GT - 1) / GT;
    if (q >= q1 + q2) return false;
    grp = q >= q1;
    i0 = grp ? n1 + (q - q1) * GT : q * GT;
    n = min(GT, (grp ? n1 + n2 : n1) - i0);
    return true;
}

// Y[(joint, item)][a][j] = sum_t Z[a][g(j) kT + t] W[T_g(j) t][j] (2 kT rows).
template <class T>
__global__ void __launch_bounds__(256) joint_rows(Geometry g, const Joint* joints, int items, int kT, const T* A,
                                                  const T* Z, T* Y) {
    __shared__ T As[GK][GT + 1], Bs[GK][GT + 1];
    const int mi = blockIdx.z, N = g.N, b = g.L * g.B, k2 = 2 * kT, it = mi % items;
    const Joint jt = joints[mi / items];
    int j0, nj, grp;
    if (!joint_tile((jt.ym - jt.y0) * b, (jt.y1 - jt.ym) * b, blockIdx.x, j0, nj, grp)) return;
    const int a0 = blockIdx.y * GT;
    const T* W = A + (size_t)it * N * N + jt.y0 * b + j0;
    const T* Zm = Z + (size_t)mi * k2 * k2 + grp * kT;
    T acc[4][4];
    tile_product<T>(kT, acc, As, Bs,
                    [&](int r, int t) { return a0 + r < k2 ? Zm[(size_t)(a0 + r) * k2 + t] : Sc<T>::zero(); },
                    [&](int t, int c) {
                        int l, p;
                        return c < nj ? W[(size_t)joint_majorana(g, jt, grp, t, l, p) * N + c] : Sc<T>::zero();
                    });
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int a = a0 + ty + 16 * u, c = tx + 16 * v;
            if (a < k2 && c < nj) Y[((size_t)it * k2 + a) * N + jt.y0 * b + j0 + c] = acc[u][v];
        }
}

// W[i][j] = (same group ? W : 0) - sum_t P[i][t] Y[g(i) kT + t][j] on tiles with
// tile(i) <= tile(j), and the negative transpose below the diagonal.
template <class T>
__global__ void __launch_bounds__(256) joint_update(Geometry g, const Joint* joints, int items, int kT, T* A, const T* P,
                                                    const T* Y) {
    __shared__ T As[GK][GT + 1], Bs[GK][GT + 1];
    if (blockIdx.y > blockIdx.x) return;
    const int mi = blockIdx.z, N = g.N, b = g.L * g.B, k2 = 2 * kT, it = mi % items;
    const Joint jt = joints[mi / items];
    const int n1 = (jt.ym - jt.y0) * b, n2 = (jt.y1 - jt.ym) * b, base = jt.y0 * b;
    int i0, ni, gi, j0, nj, gj;
    if (!joint_tile(n1, n2, blockIdx.y, i0, ni, gi) || !joint_tile(n1, n2, blockIdx.x, j0, nj, gj)) return;
    const T* Pm = P + ((size_t)it * N + base + i0) * kT;
    const T* Ym = Y + ((size_t)it * k2 + gi * kT) * N + base + j0;
    T acc[4][4];
    tile_product<T>(kT, acc, As, Bs, [&](int r, int t) { return r < ni ? Pm[(size_t)r * kT + t] : Sc<T>::zero(); },
                    [&](int t, int c) { return c < nj ? Ym[(size_t)t * N + c] : Sc<T>::zero(); });
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T* W = A + (size_t)it * N * N;
    const bool mirror = blockIdx.x != blockIdx.y, same = gi == gj;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = ty + 16 * u, c = tx + 16 * v;
            if (r >= ni || c >= nj) continue;
            const int i = base + i0 + r, j = base + j0 + c;
            T* w = W + (size_t)i * N + j;
            T x = -acc[u][v];
            if (same) x += *w;
            *w = x;
            if (mirror) W[(size_t)j * N + i] = -x;
        }
}

// ---- refinement ---------------------------------------------------------------

constexpr int RB = 8, RT = 256, MAXC = 64;

// -R = M W - I of items with act != 0 as FP32 V^T panels (rows q0 .. q0 + 7),
// the largest |R| into rmax[item]; sums in FP64.
template <class T>
__global__ void __launch_bounds__(RT) resid64(DevConst dc, const void* links, const int* cfgs, const int* pairs,
                                              const int* act, const T* A, float* Pan, size_t NK, int NP,
                                              unsigned* rmax) {
    constexpr bool CPLX = Sc<T>::CPLX;
    __shared__ int cols[MAXC];
    __shared__ T coef[RB][MAXC];
    __shared__ int ncol;
    __shared__ float red[RT / 32];
    const Geometry& g = dc.g;
    const int N = g.N, B = g.B, item = blockIdx.y;
    if (!act[item]) return;
    const T* W = A + (size_t)item * N * N;
    float* Vt = Pan + ((size_t)item * 2 + 1) * (CPLX ? 2 : 1) * NK;
    const int q0 = blockIdx.x * RB;
    if (threadIdx.x == 0) {
        // the site of q0 .. q0 + 7, then the partner ends of their links
        int n = 0;
        const int s = q0 / B;
        for (int k = 0; k < B; ++k) cols[n++] = s * B + k;
        for (int e0 = 0; e0 < RB; e0 += g.h2) {
            const int e = ((q0 + e0) % B) / g.h2, d = e >> 1, x = s % g.L, y = s / g.L;
            int ps;
            if (e & 1) ps = d == 0 ? y * g.L + (x + 1) % g.L : ((y + 1) % g.L) * g.L + x;
            else ps = d == 0 ? y * g.L + (x + g.L - 1) % g.L : ((y + g.L - 1) % g.L) * g.L + x;
            for (int k = 0; k < g.h2; ++k) {
                const int c = ps * B + (e ^ 1) * g.h2 + k;
                bool dup = false;
                for (int z = 0; z < n; ++z) dup |= cols[z] == c;
                if (!dup) cols[n++] = c;
            }
        }
        ncol = n;
    }
    __syncthreads();
    const int nc = ncol;
    for (int e = threadIdx.x; e < RB * nc; e += RT)
        coef[e / nc][e % nc] = assemble_elem<T>(dc, links, cfgs[item], pairs[item], q0 + e / nc, cols[e % nc]);
    __syncthreads();
    float mx = 0.f;
    for (int j = threadIdx.x; j < N; j += RT) {
        T acc[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) acc[r] = q0 + r == j ? -Sc<T>::one() : Sc<T>::zero();
        for (int c = 0; c < nc; ++c) {
            const T w = W[(size_t)cols[c] * N + j];
#pragma unroll
            for (int r = 0; r < RB; ++r) mac(acc[r], coef[r][c], w);
        }
        float re[RB], im[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const cxd v = Sc<T>::to(acc[r]);
            re[r] = (float)v.x;
            im[r] = (float)v.y;
            const float m = fmaxf(fabsf(re[r]), fabsf(im[r]));
            mx = (re[r] == re[r] && im[r] == im[r]) ? fmaxf(mx, m) : __int_as_float(0x7f800000);
        }
        float* dst = Vt + pidx(j, q0, NP);
        *(float4*)dst = make_float4(re[0], re[1], re[2], re[3]);
        *(float4*)(dst + 4) = make_float4(re[4], re[5], re[6], re[7]);
        if (CPLX) {
            *(float4*)(dst + NK) = make_float4(im[0], im[1], im[2], im[3]);
            *(float4*)(dst + NK + 4) = make_float4(im[4], im[5], im[6], im[7]);
        }
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int w = 0; w < RT / 32; ++w) m = fmaxf(m, red[w]);
        atomicMax(rmax + item, __float_as_uint(m));
    }
}

// U panels = W in FP32.
template <class T>
__global__ void upanel64(int N, const int* act, const T* A, float* Pan, size_t NK, int NP) {
    constexpr bool CPLX = Sc<T>::CPLX;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, q0 = blockIdx.y * 8, item = blockIdx.z;
    if (i >= N || !act[item]) return;
    const T* src = A + (size_t)item * N * N + (size_t)i * N + q0;
    float* dst = Pan + (size_t)item * 2 * (CPLX ? 2 : 1) * NK + pidx(i, q0, NP);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const cxd v = Sc<T>::to(src[t]);
        dst[t] = (float)v.x;
        if (CPLX) dst[NK + t] = (float)v.y;
    }
}

// W += W R (the FP32 product) of items with act != 0.
template <class T>
__global__ void add_product(size_t NN, const int* act, const float* D, T* A) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NN || !act[blockIdx.y]) return;
    T& a = A[blockIdx.y * NN + e];
    if constexpr (Sc<T>::CPLX) {
        const float2 d = ((const float2*)D)[blockIdx.y * NN + e];
        a = {a.x + (double)d.x, a.y + (double)d.y};
    } else {
        a += (double)D[blockIdx.y * NN + e];
    }
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

// Joints level by level: neighbouring groups of rows in pairs, an odd group
// waits; the last joint closes the torus.
std::vector<std::vector<Joint>> plan_joints(int L) {
    std::vector<int> edge(L + 1);
    for (int y = 0; y <= L; ++y) edge[y] = y;
    std::vector<std::vector<Joint>> levels;
    while (edge.size() > 2) {
        std::vector<Joint> lv;
        std::vector<int> next{0};
        size_t k = 0;
        for (; k + 2 < edge.size(); k += 2) {
            lv.push_back({edge[k], edge[k + 1], edge[k + 2], edge[k] == 0 && edge[k + 2] == L});
            next.push_back(edge[k + 2]);
        }
        if (k + 1 < edge.size()) next.push_back(edge[k + 1]);
        levels.push_back(lv);
        edge = next;
    }
    return levels;
}

constexpr int MAX_JOINTS = 32;      // of one level (L <= 64)

// Workspace of a batch: bytes per item of each array.
struct InvPlan {
    size_t a, rows, tmp, small, delta, cols, rws, prod, pan, ps, det, ints;
    size_t total(int n) const {
        return up256(a * n) + up256(rows * n) + up256(tmp * n + 4096) + 2 * up256(small * n) + up256(delta * n) +
               up256(cols * n) + up256(rws * n) + up256(prod * n) + up256(pan * n) + up256(ps * n) + up256(det * n) +
               4 * up256(ints * n) + up256(MAX_JOINTS * sizeof(Joint));
    }
};

InvPlan plan_sizes(ggf_ctx* ctx, bool cplx) {
    const Geometry& g = ctx->g;
    const size_t elem = cplx ? sizeof(cxd) : sizeof(double), N = g.N, LH = (size_t)g.L * g.h2, L = g.L;
    InvPlan p;
    p.a = N * N * elem;
    p.rows = N * L * g.B * elem;
    p.tmp = ggf_factor_tmp_bytes(g.L * g.B, g.L) + ggf_factor_tmp_bytes(2 * (int)LH, g.L) + ggf_factor_tmp_bytes(4 * (int)LH, 1);
    p.small = std::max(L / 2 * 4 * LH * LH, 16 * LH * LH) * elem;
    p.delta = std::max(L / 2 * L, 2 * L) * g.r * g.r * elem;
    p.cols = N * 2 * LH * elem;
    p.rws = 4 * LH * N * elem;
    p.prod = N * N * elem / 2;
    p.pan = panel_plane(g.N, g.N) * (cplx ? 4 : 2) * sizeof(float);
    p.ps = ggf_flush_ps_item_bytes(ctx, cplx);
    p.det = L * sizeof(cxd);
    p.ints = sizeof(int);
    return p;
}

template <class T>
ggf_status inverse_batch(ggf_ctx* ctx, const InvPlan& pl, int n, const int* cfg, const int* pair, const void* d_links,
                         std::vector<char>& ok, T** result, int** dev_cfg, int** dev_pair, cudaStream_t st) {
    constexpr bool CPLX = Sc<T>::CPLX;
    const Geometry& g = ctx->g;
    const int N = g.N, L = g.L, b = L * g.B, LH = L * g.h2;
    const size_t NN = (size_t)N * N;
    unsigned char* q = (unsigned char*)ctx->work;
    auto take = [&](size_t bytes) { unsigned char* p = q; q += up256(bytes); return p; };
    T* A = (T*)take(pl.a * n);
    T* Rb = (T*)take(pl.rows * n);
    void* tmp = take(pl.tmp * n + 4096);
    T* S = (T*)take(pl.small * n);
    T* Z = (T*)take(pl.small * n);
    T* D = (T*)take(pl.delta * n);
    T* P = (T*)take(pl.cols * n);
    T* Y = (T*)take(pl.rws * n);
    float* prod = (float*)take(pl.prod * n);
    float* Pan = (float*)take(pl.pan * n);
    unsigned char* ps = take(pl.ps * n);
    int* d_cfg = (int*)take(pl.ints * n);
    int* d_pair = (int*)take(pl.ints * n);
    int* d_act = (int*)take(pl.ints * n);
    unsigned* d_rmax = (unsigned*)take(pl.ints * n);
    Joint* d_joint = (Joint*)take(MAX_JOINTS * sizeof(Joint));
    cxd* d_det = (cxd*)take(pl.det * n);
    GGF_CK(cudaMemcpyAsync(d_cfg, cfg, n * sizeof(int), cudaMemcpyHostToDevice, st));
    GGF_CK(cudaMemcpyAsync(d_pair, pair, n * sizeof(int), cudaMemcpyHostToDevice, st));
    const DevConst dc = ctx->dc();
    const unsigned rg = (unsigned)((b * b + 255) / 256);
    row_blocks<T><<<dim3(rg, n * L), 256, 0, st>>>(dc, d_cfg, d_pair, d_links, Rb);
    GGF_TRY(ggf_invert_batched(ctx, CPLX, b, n * L, Rb, d_det, tmp, st));
    place_rows<T><<<dim3(rg, n * L), 256, 0, st>>>(N, b, L, Rb, A);
    GGF_CK(cudaGetLastError());
    ctx->launches += 2;
    for (const std::vector<Joint>& lv : plan_joints(L)) {
        const int m = (int)lv.size(), mi = m * n, cyc = lv[0].cyc, kT = LH * (cyc ? 2 : 1), nlk = L * (cyc ? 2 : 1), k2 = 2 * kT;
        int rows = 0;
        for (const Joint& j : lv) rows = std::max(rows, (j.y1 - j.y0) * b);
        int tiles = 0;
        for (const Joint& j : lv)
            tiles = std::max(tiles, ((j.ym - j.y0) * b + GT - 1) / GT + ((j.y1 - j.ym) * b + GT - 1) / GT);
        GGF_CK(cudaMemcpyAsync(d_joint, lv.data(), m * sizeof(Joint), cudaMemcpyHostToDevice, st));
        const unsigned sg = (unsigned)((k2 * k2 + 255) / 256);
        joint_delta<T><<<dim3((nlk * g.r * g.r + 127) / 128, mi), 128, 0, st>>>(dc, d_joint, n, d_cfg, d_pair, d_links, nlk, D);
        joint_small<T><<<dim3(sg, mi), 256, 0, st>>>(g, d_joint, n, kT, nlk, A, D, S);
        GGF_TRY(ggf_invert_batched(ctx, CPLX, k2, mi, S, d_det, tmp, st));
        joint_z<T><<<dim3(sg, mi), 256, 0, st>>>(g, d_joint, n, kT, nlk, S, D, Z);
        joint_cols<T><<<dim3((unsigned)(((size_t)rows * kT + 255) / 256), mi), 256, 0, st>>>(g, d_joint, n, kT, A, P);
        joint_rows<T><<<dim3(tiles, (k2 + GT - 1) / GT, mi), 256, 0, st>>>(g, d_joint, n, kT, A, Z, Y);
        joint_update<T><<<dim3(tiles, tiles, mi), 256, 0, st>>>(g, d_joint, n, kT, A, P, Y);
        GGF_CK(cudaGetLastError());
        ctx->launches += 6;
    }
    // refine while it helps: the FP64 floor of R is a few 1e-16 of |M| |W|
    const size_t NK = panel_plane(N, N);
    const int NP = panel_rows(N);
    std::vector<int> act(n, 1), pend(n);
    std::vector<float> r(n), before(n, INFINITY);
    ok.assign(n, 0);
    for (int step = 0;; ++step) {
        GGF_CK(cudaMemcpyAsync(d_act, act.data(), n * sizeof(int), cudaMemcpyHostToDevice, st));
        GGF_CK(cudaMemsetAsync(d_rmax, 0, n * sizeof(unsigned), st));
        resid64<T><<<dim3(N / RB, n), RT, 0, st>>>(dc, d_links, d_cfg, d_pair, d_act, A, Pan, NK, NP, d_rmax);
        GGF_CK(cudaGetLastError());
        GGF_CK(cudaMemcpyAsync(r.data(), d_rmax, n * sizeof(float), cudaMemcpyDeviceToHost, st));
        GGF_CK(cudaStreamSynchronize(st));
        int steps = 0;
        for (int i = 0; i < n; ++i) {
            if (!act[i]) continue;
            // at the floor, or no longer shrinking: done, if it is near enough
            const bool more = r[i] > 1e-15f && r[i] <= 1e-2f && r[i] < 0.25f * before[i] && step < 3;
            if (!more) {
                ok[i] = r[i] <= 1e-12f;
                act[i] = 0;
            }
            before[i] = r[i];
            steps += act[i];
        }
        if (steps == 0) break;
        for (int i = 0; i < n; ++i) pend[i] = act[i] ? N / 8 : 0;
        GGF_CK(cudaMemcpyAsync(d_act, pend.data(), n * sizeof(int), cudaMemcpyHostToDevice, st));
        GGF_CK(cudaMemsetAsync(prod, 0, pl.prod * n, st));
        upanel64<T><<<dim3((N + 255) / 256, N / 8, n), 256, 0, st>>>(N, d_act, A, Pan, NK, NP);
        GGF_TRY(ggf_flush_tc_items(ctx, CPLX, n, prod, nullptr, Pan, d_act, 3, ps, st));
        add_product<T><<<dim3((unsigned)((NN + 255) / 256), n), 256, 0, st>>>(NN, d_act, prod, A);
        GGF_CK(cudaGetLastError());
        ctx->launches += 5;
    }
    *result = A;
    *dev_cfg = d_cfg;
    *dev_pair = d_pair;
    return GGF_OK;
}

}  // namespace

// Whether this problem's inverses go along the lattice: below four rows the
// dense elimination has about as few steps.
bool ggf_lattice_inverse_use(const ggf_ctx* ctx) { return ctx->g.L >= 4 && ctx->use_tc && ctx->g.N % 8 == 0; }

// Matrices per batch within `budget` bytes of workspace (0: not even one), and
// the workspace they need.
int ggf_lattice_inverse_plan(ggf_ctx* ctx, bool cplx, int items, size_t budget, size_t& bytes) {
    const InvPlan p = plan_sizes(ctx, cplx);
    int n = (int)std::min<size_t>({budget / p.total(1), (size_t)items, (size_t)(65535 / std::max(ctx->g.L, 1))});
    while (n > 1 && p.total(n) > budget) --n;
    bytes = n > 0 ? p.total(n) : 0;
    return n;
}

// Inverses of n (configuration, pair) items of one family into the workspace
// (*result, item-major, with the items' device lists); ok[i] = 0 where the
// dense elimination is needed.
ggf_status ggf_lattice_inverse(ggf_ctx* ctx, bool cplx, int n, const int* cfg, const int* pair, const void* d_links,
                               std::vector<char>& ok, void** result, int** dev_cfg, int** dev_pair, cudaStream_t st) {
    const InvPlan p = plan_sizes(ctx, cplx);
    if (cplx) return inverse_batch<cxd>(ctx, p, n, cfg, pair, d_links, ok, (cxd**)result, dev_cfg, dev_pair, st);
    return inverse_batch<double>(ctx, p, n, cfg, pair, d_links, ok, (double**)result, dev_cfg, dev_pair, st);
}
