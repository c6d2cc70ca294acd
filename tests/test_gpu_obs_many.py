"""Observables of so many chains that the pair weights are formed once per chain
ahead of the kernels: the same numbers as for a few of the chains, whose CTAs
form them, and no cost that a chain's site or link pays once more."""
import numpy as np
import pytest
import torch

import ggf_inputs as gi
from tests.gpu_util import ctx_for

pytestmark = pytest.mark.gpu


def observables(p, links, precision):
    ctx = ctx_for(p)
    ctx.chains_init(links, precision=precision, refresh_every=10**9, seed=1, delay=1)
    site, link = ctx.chains_fermion()
    out = [ctx.chains_electric(), site, link, ctx.chains_fermion4(), ctx.chains_score(), ctx.chains_link_score()]
    ctx.close()
    return out


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("group,L,n_v,K,n", [
    (gi.Z2, 3, 1, 1, 700),      # one lane per chain forms its weights
    (gi.U1, 2, 2, 2, 1030),     # four lanes, three of them with a pair
    (gi.SU2, 2, 2, 4, 1030),    # sixteen lanes, ten pairs
    (gi.U1, 2, 1, 8, 1100),     # 36 pairs: more than a warp's lanes
])
def test_many_chains_as_few(group, L, n_v, K, n, precision):
    p = gi.make_problem(L, group, n_v, K, bond_scale=0.2)
    links = gi.random_links(p, n, seed=7)
    many = observables(p, links, precision)
    some = [0, 1, n // 2, n - 1]
    few = observables(p, np.ascontiguousarray(links[some]), precision)
    for a, b in zip(many, few):
        assert np.isfinite(b).all()
        assert np.array_equal(a[some], b)


def test_site_scores_of_many_chains_cost_less_than_the_electric_observable():
    """Site scores read an 8 x 8 block per site once; the electric observable reads
    as much per link, of which there are two per site, and multiplies."""
    p = gi.make_problem(8, gi.Z2, 1, 1, bond_scale=0.05)
    ctx = ctx_for(p)
    ctx.chains_init(gi.random_links(p, 1024, seed=1), precision=1, refresh_every=10**9, seed=1, delay=1)
    e = torch.zeros((1024, p.n_links, 2), dtype=torch.float64, device="cuda")
    s = torch.zeros((1024, p.V, 8, 8), dtype=torch.float64, device="cuda")

    def us(f):
        f()
        best = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                f()
            b.record()
            torch.cuda.synchronize()
            best.append(a.elapsed_time(b) / 20 * 1e3)
        return sorted(best)[2]

    # 44 and 98 us; 320 and 148 with the weights formed by every site's CTA
    assert us(lambda: ctx.chains_score(s)) < us(lambda: ctx.chains_electric(e))
    ctx.close()
