// The observable kernels' items on the host: the phases of ggf_obs_group.cuh,
// one lane after the other in place of a warp's lanes between barriers.  For
// tests that check the kernels' arithmetic and indices without a GPU; the
// kernels include ggf_obs_group.cuh itself.  Not covered here are the shuffles,
// the pair weights' warp sum and the dealing of items to blocks.
#pragma once
#include "ggf_obs_group.cuh"

namespace {

// The pairs' weights (warp_weights).
inline void item_weights(const DevConst& dc, const cxd* el, PairWeights& pw) {
    double amax, iden;
    pair_scale(dc, el, amax, iden);
    for (int p = 0; p < dc.P; ++p) {
        pw.np[p] = pair_norm(dc, el, p, amax, iden);
        pw.E[p] = dc.w[p] * pw.np[p];
    }
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
    for (int lane = 0; lane < 2; ++lane) v[lane] = electric_value<T, H, FIELD>(dc.g, lane, sh);
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
    const double gval = electric_link(g, links, c, l);
    for (int mode = 0; mode < electric_modes(g); ++mode) electric_twist<H>(g, links, c, l, mode, sh);
    PairWeights pw;
    cxd num[2] = {{0.0, 0.0}, {0.0, 0.0}};
    item_weights(dc, ell + (size_t)c * dc.P, pw);
    cxd* po = pair_out ? pair_out + ((size_t)c * g.n_links + l) * K * K : nullptr;
    for (int p = 0; p < dc.P; ++p) {
        cxd v[2];
        if (p >= K) electric_pair_item<CW, H, FIELD>(dc, p - K, l, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, gval, sh, v);
        else electric_pair_item<RW, H, FIELD>(dc, p, l, Wr + ((size_t)c * K + p) * NN, gval, sh, v);
        for (int lane = 0; lane < 2; ++lane) electric_term(dc, p, lane, true, pw.np[p], pw.E[p], v[lane], num[lane], po);
    }
    if (out) out[(size_t)c * g.n_links + l] = num[0] + num[1];
}

// The sums over the group's lanes (coupled_entry, four_point_blocks).
template <class T, int BW>
void coupled_item(const DevConst& dc, const T* W, int s, int t, typename Wide<T>::Z (&X)[4]) {
    typename Wide<T>::Z x[4];
    for (int lane = 0; lane < BW; ++lane) {
        coupled_row<T, BW>(dc, W, s, t, lane, x);
        for (int k = 0; k < 4; ++k) X[k] = lane ? X[k] + x[k] : x[k];
    }
}
template <class T, int BW>
typename Wide<T>::Z coupled_item01(const DevConst& dc, const T* W, int s) {
    typename Wide<T>::Z sum = coupled_row01<T, BW>(dc, W, s, 0);
    for (int lane = 1; lane < BW; ++lane) sum = sum + coupled_row01<T, BW>(dc, W, s, lane);
    return sum;
}

template <class T, int BW>
void fermion_pair_item(const DevConst& dc, int c, int it, int p, const T* W, cxd Np, cxd E, cxd (&acc)[BW], cxd* pair_site,
                       cxd* pair_link) {
    const FermionLane f0 = fermion_lane<BW>(dc.g, dc.K, c, it, 0);
    typename Wide<T>::Z X[4];
    coupled_item<T, BW>(dc, W, f0.s, f0.t, X);
    for (int lane = 0; lane < BW; ++lane) {
        const FermionLane f = fermion_lane<BW>(dc.g, dc.K, c, it, lane);
        cxd* po = f.is_site ? pair_site : pair_link;
        fermion_term(dc, f, p, Np, E, X[lane / (BW / 4)], acc[lane], po && f.entry ? po + f.pair : nullptr);
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
    PairWeights pw;
    cxd acc[BW] = {};
    item_weights(dc, ell + (size_t)c * dc.P, pw);
    for (int p = 0; p < dc.P; ++p) {
        if (p >= K)
            fermion_pair_item<CW, BW>(dc, c, it, p, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, pw.np[p], pw.E[p], acc, pair_site,
                                      pair_link);
        else
            fermion_pair_item<RW, BW>(dc, c, it, p, Wr + ((size_t)c * K + p) * NN, pw.np[p], pw.E[p], acc, pair_site, pair_link);
    }
    for (int lane = 0; lane < BW; ++lane) {
        const FermionLane f = fermion_lane<BW>(g, K, c, it, lane);
        cxd* out = f.is_site ? site_out : link_out;
        if (out && f.entry) out[f.out] = pair_bilinear(dc, f.s, f.t, f.a, f.b, acc[lane]);
    }
}

template <class T, int BW>
void four_point_pair_item(const DevConst& dc, int p, int s, int t, const T* W, cxd Np, cxd E, cxd (&acc)[2], cxd* q) {
    typename Wide<T>::Z x[4];
    coupled_item<T, BW>(dc, W, s, t, x);
    const auto g01 = coupled_item01<T, BW>(dc, W, s), g23 = coupled_item01<T, BW>(dc, W, t);
    for (int lane = 0; lane < 2; ++lane) four_point_term(dc, p, lane, s, t, g01, g23, x, Np, E, acc[lane], q);
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
    PairWeights pw;
    cxd acc[2] = {{0.0, 0.0}, {0.0, 0.0}};
    item_weights(dc, ell + (size_t)c * dc.P, pw);
    cxd* q = pair_out ? pair_out + ((size_t)c * g.n_links + l) * K * K : nullptr;
    for (int p = 0; p < dc.P; ++p) {
        if (p >= K)
            four_point_pair_item<CW, BW>(dc, p, s, t, Wc + ((size_t)c * dc.Kc + (p - K)) * NN, pw.np[p], pw.E[p], acc, q);
        else
            four_point_pair_item<RW, BW>(dc, p, s, t, Wr + ((size_t)c * K + p) * NN, pw.np[p], pw.E[p], acc, q);
    }
    if (out) out[(size_t)c * g.n_links + l] = s == t ? cxd{-1.0, 0.0} : acc[0] + acc[1];
}

// d log N(G) / d D_s[i][j] into out[c][s][i][j] (B x B, FP64).
template <class RW, class CW>
void score_item(const DevConst& dc, int c, int s, const RW* Wr, const CW* Wc, const cxd* ell, double* out) {
    const int B = dc.g.B;
    PairWeights pw;
    item_weights(dc, ell + (size_t)c * dc.P, pw);
    double* o = out + ((size_t)c * dc.g.V + s) * B * B;
    for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j)
            o[i * B + j] = B == 8 ? score_entry<RW, CW, 8>(dc, c, s, i, j, Wr, Wc, pw.E)
                                  : score_entry<RW, CW, 16>(dc, c, s, i, j, Wr, Wc, pw.E);
}

// The score of link block l of pair p into out[c][p][l] (R x R complex).
template <class RW, class CW, int R>
void link_score_item(const DevConst& dc, int c, int p, int l, const void* links, const RW* Wr, const CW* Wc,
                     const cxd* ell, cxd* out) {
    const Geometry& g = dc.g;
    const size_t NN = (size_t)g.N * g.N;
    PairWeights pw;
    cxd w[R * R];
    double O[(R / 2) * (R / 2)];
    LinkScoreRow<R> m[32];
    item_weights(dc, ell + (size_t)c * dc.P, pw);
    const cxd f = 0.5 * pw.E[p];
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
