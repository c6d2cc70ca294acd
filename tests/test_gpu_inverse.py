"""FP64 inverses along the lattice (chain start): against the reduced matrix
D + O Gamma_X O^T of the oracle's covariances, for lattices whose rows pair up
evenly and not, orders that are no multiple of a tile, and every group."""
import numpy as np
import pytest

import ggf_inputs as gi
from oracle import weight
from tests.gpu_util import ctx_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,L,n_v,K", [
    (gi.Z2, 4, 1, 2),     # order 128, two levels of joints
    (gi.U1, 5, 1, 2),     # order 200, an odd row waits
    (gi.U1, 6, 2, 1),     # order 576
    (gi.SU2, 5, 2, 2),    # order 400, complex pair
    (gi.Z2, 7, 2, 1),     # order 784
    (gi.U1, 3, 2, 2),     # below four rows: the dense elimination
])
def test_chain_start_inverse(group, L, n_v, K):
    p = gi.make_problem(L, group, n_v, K, bond_scale=0.2)
    links = gi.random_links(p, 2, seed=3 * L + K)
    ctx = ctx_for(p)
    ctx.chains_init(links, precision=0, refresh_every=10**9, seed=1)
    _, pairs = ctx.get_constants()
    W = weight.Weights(p)
    virt = np.array([i for i in range(p.m_s * p.V) if i % p.m_s >= 2])
    D = np.zeros((p.N, p.N))
    B = 8 * n_v
    for s in range(p.V):
        D[s * B:(s + 1) * B, s * B:(s + 1) * B] = p.gamma_site[s][2:, 2:]
    O = weight.twist_matrix(p, links[1])[np.ix_(virt, virt)]
    for k, (n, m) in enumerate(pairs):
        M = D + O @ W.GX[n, m][np.ix_(virt, virt)] @ O.T
        got = ctx.chains_inverse(1, k, p.N)
        # the refinement accepts residuals up to 1e-12; ten times that for the
        # rounding of this dense product
        assert np.abs(M @ got - np.eye(p.N)).max() < 1e-11
    ctx.close()
