"""States whose pair matrix M_01 has a singular principal block (while M_01
itself is well conditioned): one bond of the second Gaussian is rotated by
exp(v_0 A_0 + v_1 A_1), and v solves Pf(block) = 0 (a complex equation in two
real unknowns) from a start near a known root."""
import copy

import numpy as np
import scipy.linalg
import scipy.optimize

import ggf_inputs as gi
from oracle import pfaffian, weight


def reduced_matrix(p, G, n, m):
    """(M_nm, D): D + O(G) Gamma_X^{nm} O(G)^T on the virtual Majoranas, and D."""
    W = weight.Weights(p)
    virt = np.array([i for i in range(p.m_s * p.V) if i % p.m_s >= 2])
    O = weight.twist_matrix(p, G)[np.ix_(virt, virt)]
    B = 8 * p.n_v
    D = np.zeros((p.N, p.N))
    for s in range(p.V):
        D[s * B:(s + 1) * B, s * B:(s + 1) * B] = p.gamma_site[s][2:, 2:]
    return D + O @ W.GX[n, m][np.ix_(virt, virt)] @ O.T, D


class Family:
    """The K = 2 problem of `seed` with link l's second bond rotated by v."""

    def __init__(self, group, L, n_v, seed, link, skip):
        self.p = gi.make_problem(L, group, n_v, 2, bond_scale=0.3, seed=seed)
        self.link = link
        rng = np.random.default_rng(seed)
        self.A = [gi._rand_antisym(rng, self.p.r, 1.0) for _ in range(2 * skip + 2)][-2:]
        if group == gi.U1:
            q = np.concatenate([self.p.q_src, -self.p.q_src])
            self.A = [gi._project_commutant(a, q) for a in self.A]

    def at(self, v):
        q = copy.copy(self.p)
        q.gamma_bond = self.p.gamma_bond.copy()
        O = scipy.linalg.expm(v[0] * self.A[0] + v[1] * self.A[1])
        q.gamma_bond[1, self.link] = O @ q.gamma_bond[1, self.link] @ O.T
        return q

    def root(self, block, start):
        """v near `start` with Pf(block(problem)) = 0."""
        def f(v):
            z = pfaffian.pfaffian(np.array(block(self.at(v)), dtype=complex))
            return [z.real, z.imag]
        s = scipy.optimize.root(f, start, method="lm")
        assert np.hypot(*f(s.x)) < 1e-11
        return s.x


def closed_sets(p):
    """Majoranas that no later site couples to, after each site in index order
    (both ends of a link together, links ascending)."""
    L, B, h2 = p.L, 8 * p.n_v, 2 * p.n_v

    def link(i):
        s, e = i // B, (i % B) // h2
        x, y, d = s % L, s // L, e >> 1
        if e & 1:
            t = y * L + (x + 1) % L if d == 0 else ((y + 1) % L) * L + x
            return 2 * s + d, max(s, t)
        t = y * L + (x - 1) % L if d == 0 else ((y - 1) % L) * L + x
        return 2 * t + d, max(s, t)

    out = [[] for _ in range(p.V)]
    for i in range(p.N):
        out[link(i)[1]].append(i)
    return [sorted(c, key=lambda i: (link(i)[0], i)) for c in out]
