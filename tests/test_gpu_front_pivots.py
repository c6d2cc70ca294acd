"""Pivots of the site-by-site log-Pfaffian where a part of a closed set is
singular.  The closed set of the last site holds four links (n_v = 2: 32
Majoranas), which are eliminated sixteen at a time; here the first sixteen are
singular by themselves, or nearly so, and the whole set is not."""
import numpy as np
import pytest

import ggf_inputs as gi
from oracle import pfaffian
from tests.gpu_util import ctx_for, phase_dist
from tests.singular_util import Family, closed_sets, reduced_matrix

pytestmark = pytest.mark.gpu


def log_pf(p, G):
    M, _ = reduced_matrix(p, G, 0, 1)
    mag, phase = pfaffian.log_pfaffian(M)
    return mag, np.angle(phase), np.linalg.cond(M)


@pytest.mark.parametrize("offset", [0.0, 1e-8, 1e-7])
@pytest.mark.parametrize("group,L,seed,link,skip,start", [
    (gi.U1, 2, 0, 3, 0, (1.02733961, -1.02896292)),
    (gi.Z2, 2, 0, 3, 0, (1.51650408, -1.25837349)),
    (gi.Z2, 3, 1, 15, 0, (1.40553701, 1.89659374)),
    (gi.U1, 3, 0, 15, 1, (-0.67739761, 0.77071159)),
])
def test_singular_part_of_a_closed_set(group, L, seed, link, skip, start, offset):
    fam = Family(group, L, 2, seed, link, skip)
    links = gi.random_links(fam.p, 1, seed=seed)
    sets = closed_sets(fam.p)
    part = sorted(sum(sets[:-1], []) + sets[-1][:16])
    v = fam.root(lambda q: reduced_matrix(q, links[0], 0, 1)[0][np.ix_(part, part)], start)
    p = fam.at(v + np.array([offset, 0.0]))
    mag, ang, cond = log_pf(p, links[0])
    ctx = ctx_for(p)
    ctx.chains_init(links, precision=0, refresh_every=10**9, seed=1)
    ell = ctx.chains_ell()[0, 2]
    st = ctx.chains_stats()
    ctx.close()
    # the closed set has usable pivots: nothing is left to the dense elimination
    assert st.dense_pfaffians == 0
    # a backward-stable elimination of order N: N eps cond(M)
    bound = p.N * 2.2e-16 * cond
    assert abs(ell.real - mag) <= bound
    assert phase_dist(ell.imag, ang) <= bound
