"""Immediate link steps on lattices of both kinds (rows and columns copied
beside the Pfaffian, or after the decision): the cost of a rejected proposal
does not grow with the lattice, and both ways give the batched sweep's chain."""
import numpy as np
import pytest

import ggf_inputs as gi
from tests.gpu_util import ctx_for

pytestmark = pytest.mark.gpu


def rejected_link_us(L):
    """Microseconds per link of a chain whose proposals are all rejected (every
    W_SS holds a NaN: the ratio is 0)."""
    from paper_2412_01737_gb300 import ggf
    p = gi.make_problem(L, gi.U1, 2, 2, bond_scale=0.05)
    ctx = ctx_for(p)
    ctx.chains_init(gi.random_links(p, 1, seed=3), precision=0, refresh_every=10**9, seed=5, delay=1)
    B, h2 = 8 * p.n_v, 2 * p.n_v
    for pair in range(3):
        for l in range(p.n_links):
            a0 = (l >> 1) * B + (2 * (l & 1) + 1) * h2
            ctx.debug_poison_inverse(0, pair, a0, a0 + 1)
    ctx.sample_no_obs(2)
    ctx.sync()
    before = ctx.chains_stats().accepts
    ctx.profile(True)
    ctx.sample_no_obs(4)
    ctx.sync()
    ms, n = ctx.kernel_time(ggf.KT_RATIO)
    assert ctx.chains_stats().accepts == before and n == 4 * p.n_links
    ctx.close()
    return 1e3 * ms / n


def test_rejected_proposal_does_not_pay_for_the_lattice():
    # the same work per link at both sizes; copying the rows and columns of every
    # proposal takes 139 us at 12 x 12 against 48 at 4 x 4
    assert rejected_link_us(12) < 2.0 * rejected_link_us(4)


@pytest.mark.parametrize("group,L,n_v,K,precision", [
    (gi.U1, 5, 2, 2, 0),      # order 400: the complex pair's CTA copies early, the real ones' does not
    (gi.U1, 6, 2, 2, 0),      # order 576: neither
    (gi.U1, 4, 2, 2, 0),      # order 256: both, at the line
    (gi.Z2, 10, 1, 1, 0),     # order 800, one pair in FP64: just beyond it
    (gi.U1, 3, 1, 8, 0),      # 36 pairs: no spare warp
])
def test_both_ways_follow_the_batches(group, L, n_v, K, precision):
    p = gi.make_problem(L, group, n_v, K, bond_scale=0.2)
    start = gi.random_links(p, 2, seed=11)
    out = []
    for delay in (1, 8):
        ctx = ctx_for(p)
        ctx.chains_init(start, precision=precision, refresh_every=10**9, seed=31, delay=delay)
        ctx.sample(1)
        st = ctx.chains_stats()
        out.append((ctx.chains_links().copy(), ctx.chains_ell(), st.accepts))
        ctx.close()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][2] == out[1][2]
    assert np.abs(out[0][1] - out[1][1]).max() < 1e-8      # as the FP64 delayed-update parity tests
