"""Ways out of the fast factorisations: log-Pfaffians without a usable pivot,
inverses along the lattice with a singular row, and refresh batches whose
matrices need none, one and three products and the dense elimination at once;
and that ordinary states take none of them."""
import numpy as np
import pytest

import ggf_inputs as gi
from oracle import pfaffian
from tests.gpu_util import ctx_for, phase_dist
from tests.singular_util import Family, closed_sets, reduced_matrix

pytestmark = pytest.mark.gpu

PAIRS = [(0, 0), (1, 1), (0, 1)]


# ---- log-Pfaffians ---------------------------------------------------------------

@pytest.mark.parametrize("group,n_v,skip,start", [
    (gi.Z2, 1, 2, (1.35769314, 2.06122513)),
    (gi.U1, 2, 2, (0.4705153, 1.78407669)),
])
def test_singular_closed_set_goes_dense(group, n_v, skip, start):
    """All closed Majoranas after the third site of 2 x 2 singular in the complex
    pair of the middle configuration."""
    fam = Family(group, 2, n_v, 0, 1, skip)
    links = gi.random_links(fam.p, 3, seed=0)
    part = sorted(sum(closed_sets(fam.p)[:3], []))
    sub = np.ix_(part, part)
    p = fam.at(fam.root(lambda q: reduced_matrix(q, links[1], 0, 1)[0][sub], start))
    ctx = ctx_for(p)
    ell = np.zeros((3, 3, 2))
    ctx.logweight(links, ell=ell)
    ctx.chains_init(links, precision=0, refresh_every=10**9, seed=1)
    chain_ell = ctx.chains_ell()
    dense = ctx.chains_stats().dense_pfaffians
    ctx.close()
    singular = 0
    for c in range(3):
        for k, (n, m) in enumerate(PAIRS):
            M, _ = reduced_matrix(p, links[c], n, m)
            singular += np.linalg.cond(M[sub]) > 1e12
            mag, phase = pfaffian.log_pfaffian(M if n != m else M.real)
            bound = p.N * 2.2e-16 * np.linalg.cond(M)      # backward-stable eliminations of order N
            for got in (complex(*ell[c, k]), chain_ell[c, k]):
                assert abs(got.real - mag) <= bound
                assert n == m or phase_dist(got.imag, np.angle(phase)) <= bound
    assert singular >= 1 and dense == singular


# ---- FP64 inverses ---------------------------------------------------------------

def residuals(ctx, p, links):
    out = []
    for c in range(len(links)):
        for k, (n, m) in enumerate(PAIRS if p.K == 2 else [(0, 0)]):
            M, _ = reduced_matrix(p, links[c], n, m)
            W = ctx.chains_inverse(c, k, p.N)
            r = np.abs(M @ W - np.eye(p.N)).max()
            out.append(r / (p.N * 2.2e-16 * np.linalg.norm(M, 2) * np.linalg.norm(W, 2)))
    return max(out)


@pytest.mark.parametrize("group,L,n_v,K", [
    (gi.Z2, 4, 1, 2), (gi.U1, 5, 1, 2), (gi.U1, 6, 2, 1), (gi.SU2, 5, 2, 2), (gi.Z2, 7, 2, 1),
])
def test_ordinary_inverses_stay_on_the_lattice(group, L, n_v, K):
    p = gi.make_problem(L, group, n_v, K, bond_scale=0.2)
    links = gi.random_links(p, 2, seed=3 * L + K)
    ctx = ctx_for(p)
    ctx.chains_init(links, precision=0, refresh_every=10**9, seed=1)
    st = ctx.chains_stats()
    assert ctx.chains_dense_inverses() == 0 and st.dense_pfaffians == 0
    # the residual of a backward-stable inverse: N eps |M| |W|
    assert residuals(ctx, p, links) <= 1.0
    ctx.close()


@pytest.mark.parametrize("offset,dense", [(0.0, True), (1e-9, None), (1e-6, None), (1e-3, False)])
@pytest.mark.parametrize("group,L,seed,skip,start", [
    (gi.Z2, 4, 0, 1, (1.6929616, 0.04959357)),
    (gi.U1, 4, 0, 2, (0.93175598, 0.03773403)),
    (gi.Z2, 5, 1, 3, (0.98440837, 2.07562144)),
])
def test_singular_row_block(group, L, seed, skip, start, offset, dense):
    """The second row without its y links singular, or nearly so, in the complex
    pair of the middle chain: refined or inverted densely, but never worse than a
    backward-stable inverse."""
    fam = Family(group, L, 1, seed, 2 * (L + 1), skip)
    links = gi.random_links(fam.p, 3, seed=seed)
    rows = np.arange(L * 8, 2 * L * 8)
    open_ends = np.array([i for i in range(len(rows)) if (i % 8) // 2 >= 2])

    def block(q):
        M, D = reduced_matrix(q, links[1], 0, 1)
        b, d = M[np.ix_(rows, rows)].copy(), D[np.ix_(rows, rows)]
        b[open_ends, :] = d[open_ends, :]
        b[:, open_ends] = d[:, open_ends]
        return b

    p = fam.at(fam.root(block, start) + np.array([offset, 0.0]))
    ctx = ctx_for(p)
    ctx.chains_init(links, precision=0, refresh_every=10**9, seed=1)
    n = ctx.chains_dense_inverses()
    assert dense is None or (n >= 1) == dense
    assert residuals(ctx, p, links) <= 1.0
    ctx.close()


# ---- refresh of FP32 chains --------------------------------------------------------

def test_refresh_batch_of_all_kinds():
    """Inverses off by a factor 1 + x have the residual x: one batch with x
    below the FP32 floor, for one product, for three, and too large for any."""
    from paper_2412_01737_gb300 import FP32
    p = gi.make_problem(4, gi.U1, 2, 2, bond_scale=0.2)
    links = gi.random_links(p, 4, seed=3)
    ctx = ctx_for(p)
    ctx.chains_init(links, precision=FP32, refresh_every=1, seed=9, delay=1)
    for c, x in enumerate((0.0, 3e-5, 1e-3, -0.5)):
        for k in range(3):
            ctx.debug_scale_inverse(c, k, 1.0 + x)
    ctx.sample(1)
    st = ctx.chains_stats()
    assert st.refreshes == 4
    assert st.dense_refreshes == 1 and st.refine_steps >= 6 and st.max_resid > 0.05
    now = ctx.chains_links()
    for c in range(4):
        for k, (n, m) in enumerate(PAIRS):
            want = np.linalg.inv(reduced_matrix(p, now[c], n, m)[0])
            got = ctx.chains_inverse(c, k, p.N)
            assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max()    # as the refresh parity tests
    ctx.close()
