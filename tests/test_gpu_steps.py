"""Batched link steps (one cluster per chain): batches against immediate
updates, over the ways a chain's small matrices can be stored (in shared
memory, in global memory, with and without the per-batch tables) and dealt to
CTAs (one pair, two real pairs, one complex pair, several of both), and over
ragged last batches."""
import numpy as np
import pytest

import ggf_inputs as gi
from tests.gpu_util import ctx_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,L,n_v,K,delay", [
    (gi.Z2, 2, 1, 1, 3),      # one real pair, ragged batches
    (gi.Z2, 3, 1, 2, 16),     # rank 64 in two CTAs, last batch of two links
    (gi.U1, 3, 2, 2, 16),     # rank 128: FP64 matrices in global memory
    (gi.U1, 3, 1, 4, 5),      # eight CTAs
    (gi.U1, 4, 2, 1, 32),     # rank 256
    (gi.U1, 2, 1, 8, 8),      # 36 pairs: several per CTA
    (gi.U1, 4, 2, 3, 30),     # neither matrix nor tables fit in FP64
    (gi.SU2, 3, 2, 2, 7),
])
def test_batches_match_immediate_updates(group, L, n_v, K, delay):
    p = gi.make_problem(L, group, n_v, K, bond_scale=0.2)
    start = gi.random_links(p, 3, seed=17)
    out = {}
    for name, d in (("immediate", 1), ("batched", delay)):
        ctx = ctx_for(p)
        ctx.chains_init(start, precision=0, refresh_every=10**9, seed=23, delay=d)
        obs = ctx.sample(2)
        st = ctx.chains_stats()
        out[name] = (ctx.chains_links().copy(), ctx.chains_ell(), obs, st.proposals, st.accepts)
        ctx.close()
    ref, got = out["immediate"], out["batched"]
    assert np.array_equal(ref[0], got[0])
    assert ref[3:] == got[3:] and ref[3] == 3 * 2 * p.n_links
    assert np.abs(ref[1] - got[1]).max() < 1e-8      # as the FP64 delayed-update parity tests
    assert np.abs(ref[2] - got[2]).max() < 1e-8


# FP32 chains form P, Q and the next Delta beside the Pfaffian (one complex
# pair, one or two real ones per CTA) or after the decision (several pairs).
# Against the FP64 chain with the same moves: an accepted link leaves an FP32
# inverse off by at most 3.3e-6 of its largest entry (16 x 16 Z2), so 24 links
# by 8e-5; a wrong product shows at the size of the entries.
@pytest.mark.parametrize("group,L,n_v,K,delay", [
    (gi.Z2, 2, 1, 1, 3),
    (gi.Z2, 3, 1, 3, 18),     # blocks of order 4: one and two real pairs, complex ones
    (gi.U1, 3, 2, 1, 18),     # rank 144, ranks not a multiple of the warp
    (gi.U1, 3, 2, 4, 16),     # eight CTAs, ragged last batch
    (gi.U1, 2, 2, 6, 5),      # several pairs per CTA
    (gi.SU2, 3, 2, 2, 7),     # Delta of the whole batch at the start
])
def test_fp32_batches_follow_fp64(group, L, n_v, K, delay):
    p = gi.make_problem(L, group, n_v, K, bond_scale=0.05)
    start = gi.random_links(p, 2, seed=5)
    out = []
    for precision in (0, 1):
        ctx = ctx_for(p)
        ctx.chains_init(start, precision=precision, refresh_every=10**9, width=0.3, seed=29, delay=delay)
        ctx.sample(1)
        pairs = range(K * (K + 1) // 2)
        out.append((ctx.chains_links().copy(), [ctx.chains_inverse(c, q, p.N) for q in pairs for c in range(2)]))
        ctx.close()
    assert np.array_equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1], out[1][1]):
        assert np.abs(a - b).max() < 1e-3 * np.abs(a).max()
