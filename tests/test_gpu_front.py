"""Site-by-site log-Pfaffian at sizes the dense checks do not reach: fronts in
global memory and closed sets of several chunks.  log N(G) is invariant under
gauge transformations of the links, which change every entry of M."""
import numpy as np
import pytest

import ggf_inputs as gi
from tests.gpu_util import ctx_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,L,n_v,K", [
    (gi.U1, 20, 2, 2),    # 184 slots: the complex front does not fit in shared memory
    (gi.U1, 34, 2, 1),    # nor the real one
    (gi.Z2, 11, 1, 3),    # 56 slots, odd lattice
    (gi.Z2, 5, 1, 2),     # 32 slots: the small-front variant
    (gi.SU2, 7, 2, 2),
])
def test_log_weight_is_gauge_invariant(group, L, n_v, K):
    p = gi.make_problem(L, group, n_v, K)
    links = gi.random_links(p, 1, seed=5)
    rng = np.random.default_rng(9)
    if group == gi.Z2:
        h = rng.choice([-1, 1], size=p.V)
    elif group == gi.SU2:
        h = rng.normal(size=(p.V, 4))
        h /= np.linalg.norm(h, axis=1, keepdims=True)
    else:
        h = rng.uniform(0, 2 * np.pi, size=p.V)
    both = np.concatenate([links, gi.gauge_transform(p, links, h)])
    ctx = ctx_for(p)
    got = ctx.logweight(np.ascontiguousarray(both.astype(links.dtype)))
    ctx.close()
    # N/2 pivots, each to a few rounding errors of a well-conditioned front
    assert abs(got[0] - got[1]) <= 1e-10 * max(1.0, abs(got[0]))
