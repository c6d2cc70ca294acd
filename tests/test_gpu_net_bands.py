"""The network's weight gradient in bands of rows: lattices taller than one
band of shared memory, bands that do not divide the lattice, pixel counts that
are no multiple of a K step, and more work units than SMs."""
import numpy as np
import pytest

from oracle import net as onet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n", [(4, 3), (9, 2), (21, 1), (34, 2), (7, 200)])
def test_gradient_in_bands(L, n):
    from paper_2412_01737_gb300 import Net
    net = Net(0, L, 9)
    p = net.get_params()
    p[-(64 * 6 * 9 + 6):] *= 10.0        # as the whole-lattice gradient test: sharper outputs
    net.set_params(p)
    params = net.get_params().astype(np.float64)
    rng = np.random.default_rng(L)
    th = rng.uniform(0, 2 * np.pi, (n, 2 * L * L))
    bl = rng.integers(0, L, (n, 2))
    loss, g = net.loss_grad(th, bl)
    lo, go = onet.loss_and_grad(params, th, [tuple(b) for b in bl], L, quant=onet.bf16)
    net.close()
    # the bounds of the whole-lattice gradient test
    assert abs(loss - lo) <= 1e-3 * abs(lo)
    k = 0
    for ci, co in onet.LAYERS:
        m = co * ci * 9 + co
        gl, ol = g[k:k + m], go[k:k + m]
        assert np.linalg.norm(gl - ol) <= 2e-2 * np.linalg.norm(ol) + 1e-6, (ci, co)
        k += m
