// The observable kernels' items on the host: the phases of ggf_obs_group.cuh,
// one lane after the other in place of a warp's lanes between barriers.  For
// tests that check the kernels' arithmetic and indices without a GPU; the
// kernels include ggf_obs_group.cuh itself.  Not covered here are the shuffles,
// the pair weights' warp sum and the dealing of items to blocks.
#pragma once
#include "ggf_obs_group.cuh"

namespace {

// N_nm(G) / N(G) of every pair (chain_weights).
inline void item_weights(const DevConst& dc, const cxd* el, cxd* np) {
    double amax, iden;
    pair_scale(dc, el, amax, iden);
    for (int p = 0; p < dc.P; ++p) np[p] = pair_norm(dc, el, p, amax, iden);
}

template <class T, int H, bool FIELD>
void electric_pair_item(const DevConst& dc, int pf, int l, const T* W, double gval, ElectricShared<H>& sh,
                        cxd (&v)[2]) {
    constexpr int B = 4 * H;
    typename Wide<T>::Z w[B][2 * H];
    int a0, b0;
    link_ends(dc.g, l, a0, b0);
    for (int lane = 0; lane < B; ++lane) electric_load<T, H>(dc, pf, l, a0, b0, W, lane, gval, sh, w[lane]);
    for (int lane = 0; lane < B; ++lane) electric_rows<T, H>(lane, w[lane], sh);
    for (int lane = 0; lane < B; ++lane) electric_products<T, H>(dc, l, a0, lane, sh);
    for (int lane = 0; lane < 2; ++lane) v[lane] = electric_value<H, FIELD>(dc.g, lane, sh);
}

// f_E(G_c)_l into out[c][l] (if out is set) and N_nm(G) R_nm / N(G) into
// pair_out[c][l][n][m] for every ordered pair (if set).
template <class RW, class CW, int H, bool FIELD = false>
void electric_item(const DevConst& dc, int c, int l, const void* links, const RW* Wr, const CW* Wc, const cxd* ell,
                   cxd* out, cxd* pair_out) {
    const Geometry& g = dc.g;
    const int K = dc.K;
    const size_t NN = (size_t)g.N * g.N;
    ElectricShared<H> sh;
    double gval = 1.0;
    for (int lane = 0; lane < 4 * H; ++lane) gval = electric_twist<H>(g, links, c, l, lane, sh);
    cxd np[36], num[2] = {{0.0, 0.0}, {0.0, 0.0}};
    item_weights(dc, ell + (size_t)c * dc.P, np);
    cxd* po = pair_out ? pair_out + ((size_t)c * g.n_links + l) * K * K : nullptr;
    for (int p = 0; p < dc.P; ++p) {
        cxd v[2];
        if (p >= K) electric_pair_item<CW, H, FIELD>(dc, p - K, l, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, gval, sh, v);
        else electric_pair_item<RW, H, FIELD>(dc, p, l, Wr + ((size_t)c * K + p) * NN, gval, sh, v);
        for (int lane = 0; lane < 2; ++lane) electric_term(dc, p, lane, true, np[p], v[lane], num[lane], po);
    }
    if (out) out[(size_t)c * g.n_links + l] = num[0] + num[1];
}

template <class T, int BW>
void coupled_item(const DevConst& dc, const T* W, int s, int t, cxd (&X)[4]) {
    typedef typename Wide<T>::Z Z;
    Z x[BW][4];
    for (int lane = 0; lane < BW; ++lane) coupled_row<T, BW>(dc, W, s, t, lane, x[lane]);
    for (int k = 0; k < 4; ++k) {
        Z sum = x[0][k];
        for (int lane = 1; lane < BW; ++lane) sum = sum + x[lane][k];
        X[k] = as_cx(sum);
    }
}

// Item it of chain c (items 0 .. V-1 are sites, V .. V + n_links - 1 links):
// combined outputs site_out / link_out and per-pair outputs
// pair_site[c][s][n][m], pair_link[c][l][alpha][beta][n][m] =
// N_nm(G) <c c>_nm / N(G) (each may be null).
template <class RW, class CW, int BW>
void fermion_item(const DevConst& dc, int c, int it, const RW* Wr, const CW* Wc, const cxd* ell, cxd* site_out,
                  cxd* link_out, cxd* pair_site, cxd* pair_link) {
    const Geometry& g = dc.g;
    const int K = dc.K;
    const size_t NN = (size_t)g.N * g.N;
    cxd np[36], acc[4] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
    item_weights(dc, ell + (size_t)c * dc.P, np);
    for (int p = 0; p < dc.P; ++p) {
        const FermionLane f0 = fermion_lane(g, K, c, it, 0);
        cxd X[4];
        if (p >= K) coupled_item<CW, BW>(dc, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, f0.s, f0.t, X);
        else coupled_item<RW, BW>(dc, Wr + ((size_t)c * K + p) * NN, f0.s, f0.t, X);
        for (int lane = 0; lane < 4; ++lane) {
            const FermionLane f = fermion_lane(g, K, c, it, lane);
            cxd* po = f.is_site ? pair_site : pair_link;
            fermion_term(dc, f, p, np[p], X[f.a * 2 + f.b], acc[lane], po && f.entry ? po + f.pair : nullptr);
        }
    }
    for (int lane = 0; lane < 4; ++lane) {
        const FermionLane f = fermion_lane(g, K, c, it, lane);
        cxd* out = f.is_site ? site_out : link_out;
        if (out && f.entry) out[f.out] = pair_bilinear(dc, f.s, f.t, f.a, f.b, acc[lane]);
    }
}

// <c_2s c_2s+1 c_2t c_2t+1> of link l = (s -> t) of chain c into out[c][l], per
// pair into pair_out[c][l][n][m] (each may be null).
template <class RW, class CW, int BW>
void fermion4_item(const DevConst& dc, int c, int l, const RW* Wr, const CW* Wc, const cxd* ell, cxd* out,
                   cxd* pair_out = nullptr) {
    const Geometry& g = dc.g;
    const int K = dc.K;
    const size_t NN = (size_t)g.N * g.N;
    int a0, b0;
    link_ends(g, l, a0, b0);
    const int s = a0 / g.B, t = b0 / g.B;
    cxd np[36], acc[2] = {{0.0, 0.0}, {0.0, 0.0}};
    item_weights(dc, ell + (size_t)c * dc.P, np);
    cxd* q = pair_out ? pair_out + ((size_t)c * g.n_links + l) * K * K : nullptr;
    for (int p = 0; p < dc.P; ++p) {
        cxd ss[4], tt[4], x[4];
        if (p >= K) {
            const CW* W = Wc + ((size_t)c * dc.Kc + (p - K)) * NN;
            coupled_item<CW, BW>(dc, W, s, s, ss);
            coupled_item<CW, BW>(dc, W, t, t, tt);
            coupled_item<CW, BW>(dc, W, s, t, x);
        } else {
            const RW* W = Wr + ((size_t)c * K + p) * NN;
            coupled_item<RW, BW>(dc, W, s, s, ss);
            coupled_item<RW, BW>(dc, W, t, t, tt);
            coupled_item<RW, BW>(dc, W, s, t, x);
        }
        for (int lane = 0; lane < 2; ++lane) four_point_term(dc, p, lane, s, t, ss[1], tt[1], x, np[p], acc[lane], q);
    }
    if (out) out[(size_t)c * g.n_links + l] = s == t ? cxd{-1.0, 0.0} : acc[0] + acc[1];
}

// d log N(G) / d D_s[i][j] into out[c][s][i][j] (B x B, FP64).
template <class RW, class CW>
void score_item(const DevConst& dc, int c, int s, const RW* Wr, const CW* Wc, const cxd* ell, double* out) {
    const int B = dc.g.B;
    cxd np[36];
    item_weights(dc, ell + (size_t)c * dc.P, np);
    double* o = out + ((size_t)c * dc.g.V + s) * B * B;
    for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j)
            o[i * B + j] = B == 8 ? score_entry<RW, CW, 8>(dc, c, s, i, j, Wr, Wc, np)
                                  : score_entry<RW, CW, 16>(dc, c, s, i, j, Wr, Wc, np);
}

// The score of link block l of pair p into out[c][p][l] (R x R complex).
template <class RW, class CW, int R>
void link_score_item(const DevConst& dc, int c, int p, int l, const void* links, const RW* Wr, const CW* Wc,
                     const cxd* ell, cxd* out) {
    const Geometry& g = dc.g;
    const size_t NN = (size_t)g.N * g.N;
    cxd np[36], w[R * R];
    double O[(R / 2) * (R / 2)];
    LinkScoreRow<R> m[32];
    item_weights(dc, ell + (size_t)c * dc.P, np);
    const cxd f = 0.5 * (dc.w[p] * np[p]);
    for (int lane = 0; lane < 32; ++lane) {
        link_score_twist<R / 2>(dc, links, c, l, lane, O);
        if (p < dc.K) link_score_load<RW, R>(dc, Wr + ((size_t)c * dc.K + p) * NN, l, lane, w);
        else link_score_load<CW, R>(dc, Wc + ((size_t)c * dc.Kc + (p - dc.K)) * NN, l, lane, w);
    }
    for (int lane = 0; lane < 32; ++lane) link_score_mix<R>(O, w, lane, m[lane]);
    for (int lane = 0; lane < 32; ++lane) link_score_put<R>(lane, m[lane], w);
    for (int lane = 0; lane < 32; ++lane)
        link_score_out<R>(O, w, f, lane, out + (((size_t)c * dc.P + p) * g.n_links + l) * R * R);
}

}  // namespace
