"""The measured workloads of the sampler, each through the package's public
entry points, with a plain 64-bit restatement of what each one returns.

Kinds (the "kind" of a case):
  weights   log N(G) and the pair log-Pfaffians of given configurations
            (GGF.logweight): scoring configurations, checking chains
  sweep     Metropolis sweeps of resident chains (GGF.sample), then the
            configurations and log-weights a program records
  group     one sweep of several problems of uneven size (sample_group)
  energy    log N(G) and the local energy of given configurations under new
            parameters (optimize.local_energies): one evaluation of a gradient
  observe   electric, fermionic and score observables of resident chains
  train     Adam steps of the learned block proposal (Net.train)
  blocks    block moves with the learned proposal (GGF.sample_blocks)

The parameters are seeded random symmetric Gaussians: site covariances
O J O^T with O = exp(A), A normal of width 0.5 in the group's commutant, one
per sublattice; bonds maximally entangled, the further ones rotated by
generators of width 0.05 (the width at which the benchmark runs).
"""
import math

import numpy as np
import torch

from paper_2412_01737_gb300 import ggf, optimize

GROUPS = {"Z2": ggf.Z2, "U1": ggf.U1, "SU2": ggf.SU2}
WIDTH = 0.5
TWO_PI = 2.0 * math.pi


def listed():
    return [
        # every configuration of the 2x2 Z2 lattice: the smallest call, made by exhaustive sums
        {"name": "weights_z2_2x2_all", "kind": "weights", "L": 2, "group": "Z2", "n_v": 1, "K": 1, "n": 256},
        # scoring recorded configurations of the large U(1) superposition
        {"name": "weights_u1_16x16_k4", "kind": "weights", "L": 16, "group": "U1", "n_v": 2, "K": 4, "n": 16},
        # one long exact chain on the smallest lattice: launches and latency
        {"name": "chain_z2_2x2_fp64", "kind": "sweep", "L": 2, "group": "Z2", "n_v": 1, "K": 1, "n": 1,
         "precision": "FP64", "delay": 1, "refresh": 64, "sweeps": 20},
        # many small chains, rank-r update per accepted flip, frequent refresh
        {"name": "sweep_z2_8x8_fp32", "kind": "sweep", "L": 8, "group": "Z2", "n_v": 1, "K": 1, "n": 1024,
         "precision": "FP32", "delay": 1, "refresh": 64, "sweeps": 1},
        # exact double precision chains of a mid-size superposition, batched updates
        {"name": "sweep_u1_8x8_k2_fp64", "kind": "sweep", "L": 8, "group": "U1", "n_v": 2, "K": 2, "n": 24,
         "precision": "FP64", "delay": 16, "refresh": 256, "sweeps": 1},
        # the benchmark's problem with as many chains as a calibration run holds
        {"name": "sweep_u1_16x16_k4_fp32", "kind": "sweep", "L": 16, "group": "U1", "n_v": 2, "K": 4, "n": 16,
         "precision": "FP32", "delay": 16, "refresh": 2048, "sweeps": 1},
        # non-Abelian links on a lattice whose size is no multiple of any tile
        {"name": "sweep_su2_5x5_k2_fp32", "kind": "sweep", "L": 5, "group": "SU2", "n_v": 2, "K": 2, "n": 96,
         "precision": "FP32", "delay": 8, "refresh": 512, "sweeps": 1},
        # problems of uneven size, group and number of pairs swept together
        {"name": "group_uneven", "kind": "group", "cells": "8:Z2:1:64 8:U1:2:16 12:Z2:2:12 12:U1:1:6",
         "delay": 16, "refresh": 256},
        # one energy evaluation of a parameter gradient, at sampled configurations
        {"name": "energy_u1_8x8_k2", "kind": "energy", "L": 8, "group": "U1", "n_v": 2, "K": 2, "n": 8},
        # what an optimisation records of its chains after a sweep
        {"name": "observe_u1_8x8_k2", "kind": "observe", "L": 8, "group": "U1", "n_v": 2, "K": 2, "n": 32,
         "precision": "FP32"},
        # training of the proposal network on recorded configurations
        {"name": "train_16x16", "kind": "train", "L": 16, "n": 1024, "batch": 128, "steps": 8},
        # learned block moves of resident chains
        {"name": "blocks_u1_8x8_k2", "kind": "blocks", "L": 8, "group": "U1", "n_v": 2, "K": 2, "n": 32,
         "precision": "FP32", "delay": 32, "moves": 2},
    ]


def draw(rng):
    def logint(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def problem(l_lo, l_hi, k_hi, groups=("Z2", "U1", "SU2")):
        grp = rng.choice(groups)
        return {"L": logint(l_lo, l_hi), "group": grp, "n_v": 2 if grp == "SU2" else rng.choice((1, 2)),
                "K": rng.randint(1, k_hi)}

    def chains(c, most_bytes, most):
        one = pairs_bytes(c, 4)
        return max(1, min(most, int(most_bytes // one), logint(1, most)))

    kind = rng.choice(("weights", "weights", "sweep", "sweep", "sweep", "energy", "observe", "train", "blocks", "group"))
    if kind == "weights":
        c = dict(kind=kind, **problem(2, 16, 4))
        c["n"] = max(1, min(logint(1, 1024), int(2e10 // front_flops(c))))
    elif kind == "sweep":
        c = dict(kind=kind, **problem(2, 10, 4))
        c["precision"] = rng.choice(("FP64", "FP32", "FP32"))
        c["delay"] = rng.choice((1, 4, 8, 16, 16, 32))
        c["n"] = chains(c, 2**28 if c["delay"] == 1 or c["precision"] == "FP64" else 2**30, 256)
        c["refresh"] = rng.choice((64, 256, 2048))
        c["sweeps"] = 1 if c["L"] > 4 else rng.randint(1, 8)
    elif kind == "group":
        cells = []
        for _ in range(rng.randint(2, 4)):
            p = problem(3, 10, 2, ("Z2", "U1"))
            cells.append("%d:%s:%d:%d" % (p["L"], p["group"], p["K"], chains(dict(p, n_v=cell_modes(p["group"])), 2**27, 48)))
        c = {"kind": kind, "cells": " ".join(cells), "delay": rng.choice((8, 16)), "refresh": rng.choice((64, 256))}
    elif kind == "energy":
        c = dict(kind=kind, **problem(2, 8, 2, ("Z2", "U1")))
        c["n"] = chains(c, 2**26, 16)
    elif kind == "observe":
        c = dict(kind=kind, **problem(2, 8, 3))
        c.update(n=chains(c, 2**28, 48), precision=rng.choice(("FP64", "FP32")))
    elif kind == "train":
        c = {"kind": kind, "L": logint(4, 20), "n": logint(16, 2048), "batch": logint(4, 256), "steps": rng.randint(1, 8)}
    else:
        c = dict(kind=kind, **problem(4, 10, 2, ("U1",)))
        c.update(n=chains(c, 2**28, 64), precision=rng.choice(("FP64", "FP32")), delay=rng.choice((32, 36)),
                 moves=rng.randint(1, 3))
    return c


# ---- what a program has in hand -----------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "seed": seed}
    dev = torch.device("cuda", torch.cuda.current_device())
    if kind == "train":
        net = ggf.Net(dev.index, case["L"], 1)
        net.set_params(net_params(seed))
        state.update(net=net, theta=torch.from_numpy(net_data(case, seed)).to(dev))
        return state
    if kind == "group":
        state["ctxs"] = []
        for k, c in enumerate(cells_of(case)):
            ctx = context(Problem(c, seed + 31 * k), dev)
            ctx.chains_init(cold_links(c, c["n"]), precision=ggf.FP32, refresh_every=c["refresh"], width=WIDTH,
                            seed=seed + k, delay=c["delay"])
            state["ctxs"].append(ctx)
        return state
    p = Problem(case, seed)
    ctx = state["ctx"] = context(p, dev)
    if kind == "weights":
        state["links"] = torch.from_numpy(weight_links(case, seed)).to(dev)
        state["logN"] = torch.zeros(case["n"], dtype=torch.float64, device=dev)
        state["ell"] = torch.zeros(case["n"], p.P, 2, dtype=torch.float64, device=dev)
    elif kind == "energy":
        state["links"] = random_links(case, case["n"], seed)
        state["couplings"] = couplings(case)
    elif kind == "observe":
        ctx.chains_init(random_links(case, case["n"], seed), precision=getattr(ggf, case["precision"]),
                        refresh_every=1 << 30, width=WIDTH, seed=seed, delay=16)
        n, V, K, r = case["n"], p.V, p.K, p.r
        out = {"electric": (n, 2 * V, 2), "site": (n, V, 2), "link": (n, 2 * V, 2, 2, 2), "four": (n, 2 * V, 2),
               "pair_norm": (n, K, K, 2), "pair_electric": (n, 2 * V, K, K, 2), "score": (n, V, p.B, p.B),
               "link_score": (n, p.P, 2 * V, r, r, 2)}
        if case["group"] == "U1":
            out["field"] = (n, 2 * V, 2)
        state["out"] = {k: torch.zeros(s, dtype=torch.float64, device=dev) for k, s in out.items()}
    else:
        ctx.chains_init(cold_links(case, case["n"]), precision=getattr(ggf, case["precision"]),
                        refresh_every=case.get("refresh", 1 << 30), width=WIDTH, seed=seed, delay=case["delay"])
        rows = case["sweeps"] if kind == "sweep" else case["moves"]
        state["obs"] = torch.zeros(rows, case["n"], ggf.N_OBS, dtype=torch.float64, device=dev)
        state["links"] = torch.from_numpy(cold_links(case, case["n"])).to(dev)
        if kind == "blocks":
            state["net"] = ggf.Net(dev.index, case["L"], 1)
            state["net"].set_params(net_params(seed))
    return state


def context(p, dev):
    ctx = ggf.GGF(dev.index)
    ctx.init_problem(p)
    return ctx


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "weights":
        state["ctx"].logweight(state["links"], state["logN"], state["ell"])
        return {"logN": state["logN"], "ell": state["ell"]}
    if kind == "energy":
        logN, h = optimize.local_energies(state["ctx"], state["links"], **state["couplings"])
        return {"logN": logN, "h": h}
    if kind == "train":
        losses = state["net"].train(state["theta"], case["batch"], case["steps"], 2e-3)
        return {"losses": losses, "params": state["net"].get_params()}
    if kind == "group":
        obs = ggf.sample_group(state["ctxs"], 1)
        return {"obs": obs, "links": [c.chains_links() for c in state["ctxs"]],
                "ell": [c.chains_ell() for c in state["ctxs"]]}
    ctx = state["ctx"]
    if kind == "observe":
        o = state["out"]
        ctx.chains_electric(o["electric"])
        if "field" in o:
            ctx.chains_electric_field(o["field"])
        ctx.chains_fermion(o["site"], o["link"])
        ctx.chains_fermion4(o["four"])
        ctx.chains_pairs(ggf.PAIRS_NORM, o["pair_norm"])
        ctx.chains_pairs(ggf.PAIRS_ELECTRIC, o["pair_electric"])
        ctx.chains_score(o["score"])
        ctx.chains_link_score(o["link_score"])
        return dict(o)
    if kind == "blocks":
        ctx.sample_blocks(state["net"], case["moves"], state["obs"])
    else:
        ctx.sample(case["sweeps"], state["obs"])
    return {"obs": state["obs"], "links": ctx.chains_links(state["links"]), "ell": ctx.chains_ell()}


# ---- what a pass cannot do without --------------------------------------------------


def pairs_bytes(c, real):
    """Bytes of one chain's inverses (K real and K (K - 1) / 2 complex ones)."""
    N = 8 * c["n_v"] * c["L"] ** 2
    return N * N * real * (c["K"] + c["K"] * (c["K"] - 1))


def front_flops(c):
    """Elimination of one configuration's matrices along the lattice: a front
    of two rows of link ends, one rank-2 update of its triangle per pair of
    Majoranas, real pairs once and complex ones four times."""
    h2, L = 2 * c["n_v"], c["L"]
    f = min((2 * L + 1) * h2, 4 * h2 * L * L)
    return 8 * c["n_v"] * L * L * f * f * (c["K"] + 2 * c["K"] * (c["K"] - 1))


def work(case):
    kind = case["kind"]
    if kind == "group":
        parts = [work(dict(c, kind="sweep", sweeps=1, precision="FP32")) for c in cells_of(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "train":
        # per sample and layer: forward, input and weight gradient of the 3 x 3 convolutions; activations once each way
        px, macs = case["batch"] * case["L"] ** 2, 9 * (8 * 64 + 2 * 64 * 64 + 64 * 6)
        act = px * (2 * (8 + 3 * 64) + 4 * 6)
        return {"bytes": case["steps"] * (2 * act + 81990 * 4 * 6), "flops": case["steps"] * 6 * px * macs}
    n, V = case["n"], case["L"] ** 2
    N, r, K = 8 * case["n_v"] * V, 4 * case["n_v"], case["K"]
    P, mults = K * (K + 1) // 2, K + 2 * K * (K - 1)
    rows = {"Z2": 1, "U1": 8, "SU2": 32}[case["group"]] * 2 * V
    if kind == "weights":
        return {"bytes": n * (rows + 8 + 16 * P), "flops": n * front_flops(case)}
    if kind == "energy":
        # log-weights, then every entry of the inverses that the local observables read: an elimination of all columns
        return {"bytes": n * (rows + 24 + pairs_bytes(case, 8)), "flops": n * 2.0 * N * N * (2 * case["L"] + 1) * r * mults}
    if kind == "observe":
        # the site and link blocks of every inverse, and the outputs
        B = 8 * case["n_v"]
        real = 8 if case["precision"] == "FP64" else 4
        read = (K + K * (K - 1)) * real * V * 3 * B * B
        put = 16 * (2 * V * (2 + K * K) + V + 8 * V + 2 * V + K * K + P * 2 * V * r * r) + 8 * V * B * B
        return {"bytes": n * (read + put), "flops": n * V * 3 * B * B * 16.0 * mults}
    # a batch of `delay` links (immediate updates: one link) folds one update of their rank into every inverse
    real = 8 if case["precision"] == "FP64" else 4
    if kind == "blocks":
        return {"bytes": case["moves"] * n * 2.0 * pairs_bytes(case, real), "flops": case["moves"] * n * 2.0 * N * N * 32 * r * mults}
    batches = math.ceil(2 * V / case["delay"])
    return {"bytes": case["sweeps"] * n * 2.0 * pairs_bytes(case, real) * batches,
            "flops": case["sweeps"] * n * 2.0 * N * N * 2 * V * r * mults}


# ---- inputs -------------------------------------------------------------------------


def cell_modes(group):
    return 1 if group == "Z2" else 2


def cells_of(case):
    out = []
    for cell in case["cells"].split():
        L, grp, K, n = cell.split(":")
        out.append({"L": int(L), "group": grp, "n_v": cell_modes(grp), "K": int(K), "n": int(n),
                    "delay": case["delay"], "refresh": case["refresh"]})
    return out


def vacuum(modes):
    return np.kron(np.eye(modes), np.array([[0.0, -1.0], [1.0, 0.0]]))


def expm(A):
    return torch.linalg.matrix_exp(torch.from_numpy(A)).numpy()


def quat_rotation(q):
    """Majorana rotations (..., 4, 4) of the doublet twist of unit quaternions (..., 4)."""
    a0, a1, a2, a3 = (q[..., k] for k in range(4))
    # u = [[a0 + i a3, a2 + i a1], [-a2 + i a1, a0 - i a3]]
    re, im = {(0, 0): a0, (0, 1): a2, (1, 0): -a2, (1, 1): a0}, {(0, 0): a3, (0, 1): a1, (1, 0): a1, (1, 1): -a3}
    R = q.new_zeros(q.shape[:-1] + (4, 4)) if torch.is_tensor(q) else np.zeros(q.shape[:-1] + (4, 4))
    for j in range(2):
        for k in range(2):
            R[..., 2 * j, 2 * k] = re[k, j]
            R[..., 2 * j, 2 * k + 1] = im[k, j]
            R[..., 2 * j + 1, 2 * k] = -im[k, j]
            R[..., 2 * j + 1, 2 * k + 1] = re[k, j]
    return R


class Problem:
    """The parameters that GGF.init_problem takes."""

    def __init__(self, case, seed):
        rng = np.random.default_rng(seed)
        self.L, self.group_name, self.n_v, self.K = case["L"], case["group"], case["n_v"], case["K"]
        self.group = GROUPS[self.group_name]
        L, n_v = self.L, self.n_v
        self.V, self.B, self.h2, self.r = L * L, 8 * n_v, 2 * n_v, 4 * n_v
        self.N, self.P = self.B * self.V, self.K * (self.K + 1) // 2
        self.q_src = np.array([1 if j % 2 == 0 else -1 for j in range(n_v)], dtype=np.int32)
        self.q_phys = np.array([(-1) ** (s % L + s // L) for s in range(self.V)], dtype=np.int32)
        ends, conj = [1] * n_v, [-1] * n_v
        src, dst = list(self.q_src), list(-self.q_src)
        kinds = {q: self._site(rng, [q] + dst + src + dst + src, [0] + conj + ends + conj + ends)
                 for q in (1, -1)}
        self.gamma_site = np.stack([kinds[int(q)] for q in self.q_phys])
        first = np.eye(self.r)
        c = math.sqrt(0.5)
        for j in range(n_v):
            for a, s in ((2 * j, c), (2 * j + 1, -c)):
                b = self.h2 + a
                first[a, a], first[a, b], first[b, a], first[b, b] = c, s, -s, c
        g1 = first @ vacuum(self.h2) @ first.T
        bonds = [g1]
        for _ in range(1, self.K):
            O = expm(self._commutant(self._antisymmetric(rng, self.r, 0.05), src + dst, ends + conj))
            bonds.append(O @ g1 @ O.T)
        self.bonds = np.stack(bonds)                       # (K, r, r), the same on every link
        self.gamma_bond = np.repeat(self.bonds[:, None], 2 * self.V, axis=1)
        z = rng.normal(size=self.K) + 1j * rng.normal(size=self.K)
        self.lam = z / np.linalg.norm(z)

    @staticmethod
    def _antisymmetric(rng, n, scale):
        X = np.triu(rng.normal(size=(n, n)) * scale, 1)
        return X - X.T

    def _commutant(self, A, charges, doublets):
        """The part of A that commutes with the group's action on modes of the
        given U(1) charges, or on SU(2) doublets (+1) and conjugate doublets
        (-1) of two consecutive modes (0: a singlet): the average over the
        group, exact over 16 angles or over the eight unit quaternions
        +-1, +-i, +-j, +-k (the entries transform with spin 0, 1/2 and 1)."""
        if self.group_name == "Z2":
            return A
        turns = []
        if self.group_name == "U1":
            for k in range(16):
                R = np.zeros_like(A)
                for j, q in enumerate(charges):
                    c, s = math.cos(q * TWO_PI * k / 16), math.sin(q * TWO_PI * k / 16)
                    R[2 * j:2 * j + 2, 2 * j:2 * j + 2] = [[c, s], [-s, c]]
                turns.append(R)
        else:
            for quat in np.concatenate([np.eye(4), -np.eye(4)]):
                R = np.eye(len(A))
                j = 0
                while j < len(doublets):
                    if doublets[j] == 0:
                        j += 1
                        continue
                    u = quat * ([1, 1, 1, 1] if doublets[j] > 0 else [1, -1, 1, -1])   # complex conjugate
                    R[2 * j:2 * j + 4, 2 * j:2 * j + 4] = quat_rotation(u)
                    j += 2
                turns.append(R)
        return sum(R.T @ A @ R for R in turns) / len(turns)

    def _site(self, rng, charges, doublets):
        O = expm(self._commutant(self._antisymmetric(rng, 2 + self.B, 0.5), charges, doublets))
        return O @ vacuum(1 + 4 * self.n_v) @ O.T


def cold_links(case, n):
    nl = 2 * case["L"] ** 2
    if case["group"] == "Z2":
        return np.ones((n, nl), dtype=np.int8)
    if case["group"] == "U1":
        return np.zeros((n, nl))
    return np.tile(np.array([1.0, 0.0, 0.0, 0.0]), (n, nl, 1))


def random_links(case, n, seed):
    rng = np.random.default_rng([seed, 1])
    nl = 2 * case["L"] ** 2
    if case["group"] == "Z2":
        return rng.choice(np.array([1, -1], dtype=np.int8), size=(n, nl))
    if case["group"] == "U1":
        return rng.uniform(0.0, TWO_PI, size=(n, nl))
    q = rng.normal(size=(n, nl, 4))
    return q / np.linalg.norm(q, axis=-1, keepdims=True)


def weight_links(case, seed):
    nl = 2 * case["L"] ** 2
    if case["group"] == "Z2" and case["n"] == 2 ** min(nl, 30):      # all of them
        return (1 - 2 * ((np.arange(case["n"])[:, None] >> np.arange(nl)) & 1)).astype(np.int8)
    return random_links(case, case["n"], seed)


def couplings(case):
    """Plaquette, electric, staggered mass and hopping terms of a lattice gauge Hamiltonian."""
    V, L = case["L"] ** 2, case["L"]
    q = np.array([(-1) ** (s % L + s // L) for s in range(V)], dtype=np.int32)
    return {"c_plaquette": -1.0, "c_electric": np.full(2 * V, 0.6), "c_site": 0.8 * q, "c_hop": np.full(2 * V, 0.5),
            "charges": q}


LAYERS = [(8, 64), (64, 64), (64, 64), (64, 6)]


def net_params(seed):
    rng = np.random.default_rng([seed, 2])
    out = []
    for k, (ci, co) in enumerate(LAYERS):
        bound = math.sqrt(6.0 / (9 * ci)) * (0.1 if k == len(LAYERS) - 1 else 1.0)
        out += [rng.uniform(-bound, bound, size=co * ci * 9), np.zeros(co)]
    return np.concatenate(out).astype(np.float32)


def net_data(case, seed):
    """Angles near the identity, as chains give them: they spread with the distance."""
    rng = np.random.default_rng([seed, 3])
    return np.mod(rng.normal(scale=0.8, size=(case["n"], 2 * case["L"] ** 2)), TWO_PI)


# ---- the same results in 64 bits ----------------------------------------------------


def exact(case, seed):
    kind = case["kind"]
    if kind == "blocks":
        return None               # the proposed angles are those of a 16-bit network
    if kind == "train":
        return exact_train(case, seed)
    if kind == "group":
        parts = [exact_sweep(Problem(c, seed + 31 * k), c, seed + k, 1) for k, c in enumerate(cells_of(case))]
        return {k: [part[k] for part in parts] for k in ("obs", "links", "ell")}
    p = Problem(case, seed)
    if kind == "sweep":
        if p.N > 2500:
            return None           # minutes in double precision
        return exact_sweep(p, case, seed, case["sweeps"])
    if kind == "weights":
        ell = log_pfaffians(p, values(p, weight_links(case, seed)))
        return {"logN": terms(p, ell)[0], "ell": torch.view_as_real(ell)}
    links = values(p, random_links(case, case["n"], seed))
    ell = log_pfaffians(p, links)
    logN, weight = terms(p, ell)
    found = observables(p, links, weight)
    if kind == "energy":
        c = couplings(case)
        h = c["c_plaquette"] * plaquettes(p, links) + found["electric"] @ cplx(c["c_electric"])
        h = h + (0.5 * (1.0 + 1j * found["site"])) @ cplx(c["c_site"])
        h = h + 2.0 * link_terms(p, links, found["link"], c["charges"]).real @ cplx(c["c_hop"]).real
        return {"logN": logN.cpu().numpy(), "h": h.cpu().numpy()}
    out = {k: torch.view_as_real(v.contiguous()) if v.is_complex() else v for k, v in found.items()}
    if case["group"] != "U1":
        del out["field"]
    return out


def device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def cplx(a):
    return torch.from_numpy(np.asarray(a, dtype=np.complex128)).to(device())


def values(p, links):
    t = torch.from_numpy(links).to(device())
    return t.double()


def pair_list(p):
    return [(n, n) for n in range(p.K)] + [(n, m) for n in range(p.K) for m in range(n + 1, p.K)]


def small_pfaffian(A):
    """Pfaffian of a small matrix (numpy, complex) by expansion along the first row."""
    n = len(A)
    if n == 0:
        return 1.0
    total = 0.0
    for j in range(1, n):
        if A[0, j] != 0:
            keep = [k for k in range(1, n) if k != j]
            total += (-1) ** (j - 1) * A[0, j] * small_pfaffian(A[np.ix_(keep, keep)])
    return total


def transition(ket, bra):
    """Covariance of |ket><bra| / <bra|ket>."""
    I = np.eye(len(ket))
    Fk, Fb = -1j * ket, -1j * bra
    return 1j * (I - (I - Fk) @ np.linalg.inv(I + Fb @ Fk) @ (I - Fb))


def permutation_sign(order):
    order, seen, cycles = list(order), [False] * len(order), 0
    for i in range(len(order)):
        if not seen[i]:
            cycles += 1
            while not seen[i]:
                seen[i] = True
                i = order[i]
    return -1 if (len(order) - cycles) % 2 else 1


def link_indices(p):
    """(2V, r) virtual Majoranas of every link: the source end, then the target end."""
    L = p.L
    l = np.arange(2 * p.V)
    s, d = l // 2, l % 2
    x, y = s % L, s // L
    t = np.where(d == 0, y * L + (x + 1) % L, ((y + 1) % L) * L + x)
    k = np.arange(p.h2)
    return np.concatenate([(s * p.B + (2 * d + 1) * p.h2)[:, None] + k, (t * p.B + 2 * d * p.h2)[:, None] + k], axis=1)


def constants(p):
    """Per pair: the link block of Gamma_X, log c and the weight in the sum
    N(G) = Re sum_p w_p exp(log c_p + log Pf M_p)."""
    half, nl, n_virt = p.r // 2, 2 * p.V, 0.5 * p.N
    sign = permutation_sign(link_indices(p).reshape(-1))

    def overlap2(a, b):
        return 2.0 ** -half * small_pfaffian(a) * small_pfaffian(a + b)

    out = []
    for n, m in pair_list(p):
        Gn, Gm, G0 = p.bonds[n].astype(complex), p.bonds[m].astype(complex), p.bonds[0].astype(complex)
        if n == m:
            out.append((Gn, -n_virt * math.log(2.0) + 0j, abs(p.lam[n]) ** 2 + 0j))
            continue
        Gx = transition(Gn, Gm)
        num = overlap2(Gm, Gn) * overlap2(G0, transition(Gm, Gn))
        ov = num / math.sqrt(overlap2(G0, Gm).real * overlap2(G0, Gn).real)
        up = (small_pfaffian(Gx) ** nl * sign).real >= 0
        lc = nl * np.log(ov) + (0.0 if up else 1j * math.pi) - n_virt * math.log(2.0)
        out.append((Gx, lc, 2.0 * np.conj(p.lam[n]) * p.lam[m]))
    return out


def twists(p, links):
    """Rotations (..., h2, h2) of the source ends for link values (..., [4])."""
    if p.group_name == "SU2":
        return quat_rotation(links)
    eye = torch.eye(p.h2, dtype=torch.float64, device=links.device)
    if p.group_name == "Z2":
        return links[..., None, None] * eye
    R = links.new_zeros(links.shape + (p.h2, p.h2))
    for j in range(p.n_v):
        c, s = torch.cos(int(p.q_src[j]) * links), torch.sin(int(p.q_src[j]) * links)
        R[..., 2 * j, 2 * j], R[..., 2 * j, 2 * j + 1] = c, s
        R[..., 2 * j + 1, 2 * j], R[..., 2 * j + 1, 2 * j + 1] = -s, c
    return R


def twisted(p, G, links):
    """O G O^T (..., r, r) for one pair's link block G."""
    h, G = p.h2, cplx(G)
    R = twists(p, links).to(torch.complex128)
    out = G.expand(R.shape[:-2] + G.shape).clone()
    out[..., :h, :] = R @ out[..., :h, :]
    out[..., :, :h] = out[..., :, :h] @ R.transpose(-1, -2)
    return out


def site_blocks(p):
    return torch.from_numpy(p.gamma_site[:, 2:, 2:].copy()).to(device())


def matrices(p, G, links):
    """(D, Gamma_tw) of M = D + Gamma_tw, dense and complex: (N, N) and (n, N, N)."""
    idx = torch.from_numpy(link_indices(p)).to(device())
    tw = torch.zeros(len(links), p.N, p.N, dtype=torch.complex128, device=device())
    tw[:, idx[:, :, None], idx[:, None, :]] = twisted(p, G, links)
    D = torch.block_diag(*site_blocks(p)).to(torch.complex128)
    return D, tw


def eliminate(A, count, logabs, phase):
    """Eliminates the first `count` rows and columns of a batch of antisymmetric
    matrices pair by pair (largest pivot of the column among them) and returns
    the Schur complement; log |Pf| and the phase are updated in place."""
    n = A.shape[-1]
    items = torch.arange(len(A), device=A.device)
    for k in range(0, count, 2):
        q = k + 1
        pick = k + 1 + A[:, k + 1:count, k].abs().argmax(dim=1)
        rows, other = A[:, q].clone(), A[items, pick].clone()
        A[:, q] = other
        A[items, pick] = rows
        cols, other = A[:, :, q].clone(), A[items, :, pick].clone()
        A[:, :, q] = other
        A[items, :, pick] = cols
        a = A[:, k, q].clone()
        logabs += a.abs().log()
        phase *= torch.where(pick == q, 1.0, -1.0) * a / a.abs()
        if q + 1 < n:
            u, v = A[:, k, q + 1:] / a[:, None], A[:, q, q + 1:]
            S = A[:, q + 1:, q + 1:]
            S += v[:, :, None] * u[:, None, :]
            S -= u[:, :, None] * v[:, None, :]
    return A[:, count:, count:]


def log_pfaffians(p, links):
    """log Pf(M_p) per configuration and pair, by eliminating the lattice row
    by row (the Majoranas whose site and link partner are both present)."""
    idx = link_indices(p)
    partner = np.zeros(p.N, dtype=np.int64)
    link_of = np.zeros((p.N, 2), dtype=np.int64)
    for l, ii in enumerate(idx):
        for pos, i in enumerate(ii):
            link_of[i] = l, pos
            partner[i] = (ii[p.h2:] if pos < p.h2 else ii[:p.h2])[0] // (p.L * p.B)
    sites, out = site_blocks(p).to(torch.complex128), []
    for (n, m), (G, _, _) in zip(pair_list(p), constants(p)):
        tw = twisted(p, G, links)
        logabs = torch.zeros(len(links), dtype=torch.float64, device=device())
        phase = torch.ones(len(links), dtype=torch.complex128, device=device())
        active, front, order = np.zeros(0, dtype=np.int64), None, []
        for y in range(p.L):
            new = np.arange(y * p.L * p.B, (y + 1) * p.L * p.B)
            have = np.concatenate([active, new])
            gone = partner[have] <= y
            have, old = np.concatenate([have[gone], have[~gone]]), len(active)
            where = {int(i): k for k, i in enumerate(have)}
            A = torch.zeros(len(links), len(have), len(have), dtype=torch.complex128, device=device())
            if old:
                at = torch.tensor([where[int(i)] for i in active], device=device())
                A[:, at[:, None], at[None, :]] = front
            for s in range(y * p.L, (y + 1) * p.L):
                at = torch.tensor([where[s * p.B + k] for k in range(p.B)], device=device())
                A[:, at[:, None], at[None, :]] += sites[s]
            fresh = set(int(i) for i in new)
            for l in sorted(set(link_of[new, 0].tolist())):
                pos = [k for k, i in enumerate(idx[l]) if int(i) in where]
                isnew = torch.tensor([int(idx[l][k]) in fresh for k in pos], device=device())
                at, ps = torch.tensor([where[int(idx[l][k])] for k in pos], device=device()), torch.tensor(pos, device=device())
                add = tw[:, l][:, ps[:, None], ps[None, :]] * (isnew[:, None] | isnew[None, :])
                A[:, at[:, None], at[None, :]] += add
            count = int(gone.sum())
            order += have[:count].tolist()
            front, active = eliminate(A, count, logabs, phase), have[count:]
        phase = phase * permutation_sign(order)
        out.append(torch.complex(logabs, torch.zeros_like(logabs) if n == m else phase.angle()))
    return torch.stack(out, dim=1)


def terms(p, ell):
    """log N(G) and N_nm(G) / N(G) per pair of `pair_list`."""
    cs = constants(p)
    logc, w = cplx([c[1] for c in cs]), cplx([c[2] for c in cs])
    e = logc + ell
    e = torch.complex(e.real, torch.where(torch.arange(p.P, device=e.device) < p.K, 0.0, e.imag))
    top = e.real.max(dim=1, keepdim=True).values
    scaled = torch.exp(e - top)
    total = (w * scaled).real.sum(dim=1)
    return top[:, 0] + total.log(), scaled / total[:, None]


def plaquettes(p, links):
    L, s = p.L, np.arange(p.V)
    x, y = s % L, s // L
    l1, l2, l3, l4 = 2 * s, 2 * (y * L + (x + 1) % L) + 1, 2 * (((y + 1) % L) * L + x), 2 * s + 1
    if p.group_name == "Z2":
        return (links[:, l1] * links[:, l2] * links[:, l3] * links[:, l4]).mean(dim=1)
    if p.group_name == "U1":
        return torch.cos(links[:, l1] + links[:, l2] - links[:, l3] - links[:, l4]).mean(dim=1)
    turn = links.new_tensor([1.0, -1.0, -1.0, -1.0])
    a, b = quat_mul(links[:, l1] * turn, links[:, l2] * turn), quat_mul(links[:, l3], links[:, l4])
    return (a * b * turn).sum(dim=-1).mean(dim=1)


def quat_mul(a, b):
    """(a0 + i a.s)(b0 + i b.s) of quaternions (..., 4)."""
    s = a[..., :1] * b[..., :1] - (a[..., 1:] * b[..., 1:]).sum(dim=-1, keepdim=True)
    v = a[..., :1] * b[..., 1:] + b[..., :1] * a[..., 1:] - torch.linalg.cross(a[..., 1:], b[..., 1:])
    return torch.cat([s, v], dim=-1)


def small_pf(G):
    return G[..., 0, 1] if G.shape[-1] == 2 else G[..., 0, 1] * G[..., 2, 3] - G[..., 0, 2] * G[..., 1, 3] + G[..., 0, 3] * G[..., 1, 2]


def electric_value(p, G, field):
    """Expectation of the link insertion from the end's covariance G (..., h2, h2)."""
    occ = [0.5 * (1.0 + G[..., 2 * j, 2 * j + 1]) for j in range(p.n_v)]
    q = [int(v) for v in p.q_src]
    if field:
        return sum(q[j] * occ[j] for j in range(p.n_v))
    if p.group_name == "Z2":
        return (-1) ** p.n_v * small_pf(G)
    both = 0.25 * (1.0 + G[..., 0, 1] + G[..., 2, 3] + small_pf(G)) if p.n_v == 2 else None
    if p.group_name == "SU2":
        return 0.75 * (occ[0] + occ[1] - 2.0 * both)
    out = sum(q[j] * q[j] * occ[j] for j in range(p.n_v))
    return out + 2 * q[0] * q[1] * both if p.n_v == 2 else out


def observables(p, links, weight):
    """Everything that local_energies and the chains' observables are made of,
    from dense inverses by Wick's theorem."""
    n, V, K, h = len(links), p.V, p.K, p.h2
    idx = torch.from_numpy(link_indices(p)).to(device())
    S, src, dst = idx[:, :h], idx[:, 0] // p.B, idx[:, h] // p.B
    sites = torch.arange(V, device=device())
    Ap = torch.block_diag(*torch.from_numpy(p.gamma_site[:, :2, :2].copy())).to(device())
    Bp = torch.block_diag(*torch.from_numpy(p.gamma_site[:, :2, 2:].copy())).to(torch.complex128).to(device())
    eye = torch.eye(p.N, dtype=torch.complex128, device=device())
    zero = lambda *s: torch.zeros((n,) + s, dtype=torch.complex128, device=device())  # noqa: E731
    out = {"electric": zero(2 * V), "field": zero(2 * V), "site": zero(V), "link": zero(2 * V, 2, 2), "four": zero(2 * V),
           "pair_norm": zero(K, K), "pair_electric": zero(2 * V, K, K),
           "score": torch.zeros(n, V, p.B, p.B, dtype=torch.float64, device=device()),
           "link_score": zero(p.P, 2 * V, p.r, p.r)}
    O = torch.zeros(n, 2 * V, p.r, p.r, dtype=torch.complex128, device=device())
    O[..., :h, :h] = twists(p, links).to(torch.complex128)
    O[..., h:, h:] = torch.eye(h, dtype=torch.complex128, device=device())
    for k, ((a, b), (G, _, w)) in enumerate(zip(pair_list(p), constants(p))):
        D, tw = matrices(p, G, links)
        W = torch.linalg.inv(D + tw)
        block = torch.arange(p.B, device=device()) + (sites * p.B)[:, None]
        Ws = W[:, block[:, :, None], block[:, None, :]]
        out["score"] += 0.5 * (w * weight[:, k, None, None, None] * Ws.transpose(-1, -2)).real
        Wl = W[:, idx[:, :, None], idx[:, None, :]]
        out["link_score"][:, k] = 0.5 * w * weight[:, k, None, None, None] * (O.transpose(-1, -2) @ Wl @ O).transpose(-1, -2)
        for turn in range(1 if a == b else 2):             # the pair's two orders
            cj = (lambda v: v.conj()) if turn else (lambda v: v)
            i, j = (b, a) if turn else (a, b)
            Np = cj(weight[:, k])
            wn = (np.conj(p.lam[i]) * p.lam[j]) * Np
            out["pair_norm"][:, i, j] = Np
            left, right = eye + 1j * D, eye + 1j * cj(tw)
            cov = 1j * eye - left @ (cj(W) @ right)
            Gs = cov[:, S[:, :, None], S[:, None, :]]
            value = electric_value(p, Gs, False)
            out["electric"] += wn[:, None] * value
            out["field"] += wn[:, None] * electric_value(p, Gs, True)
            out["pair_electric"][:, :, i, j] = Np[:, None] * value
            eff = Ap + Bp @ cj(W) @ Bp.T
            bil = -1j * eff
            out["site"] += wn[:, None] * bil[:, 2 * sites, 2 * sites + 1]
            two = torch.arange(2, device=device())
            la, lb = (2 * src)[:, None, None] + two[:, None], (2 * dst)[:, None, None] + two
            blk = bil[:, la, lb]
            same = (src == dst)[:, None, None] & (two[:, None] == two)
            out["link"] += wn[:, None, None, None] * torch.where(same, torch.ones_like(blk), blk)
            pf = eff[:, 2 * src, 2 * src + 1] * eff[:, 2 * dst, 2 * dst + 1] - eff[:, 2 * src, 2 * dst] * eff[:, 2 * src + 1, 2 * dst + 1] \
                + eff[:, 2 * src, 2 * dst + 1] * eff[:, 2 * src + 1, 2 * dst]
            out["four"] -= wn[:, None] * torch.where(src == dst, torch.ones_like(pf), pf)
    return out


def link_terms(p, links, X, charges):
    idx = link_indices(p)
    e_s = torch.from_numpy(np.where(charges[idx[:, 0] // p.B] > 0, 1.0, -1.0)).to(device())
    e_t = torch.from_numpy(np.where(charges[idx[:, p.h2] // p.B] > 0, -1.0, 1.0)).to(device())
    u = links.to(torch.complex128) if p.group_name == "Z2" else torch.exp(1j * links)
    return u * 0.25 * (X[..., 0, 0] + 1j * e_t * X[..., 0, 1] + 1j * e_s * X[..., 1, 0] - e_s * e_t * X[..., 1, 1])


def philox(counters, k0, k1):
    """Philox4x64-10 of four counter words and two keys (broadcast uint64 arrays)."""
    c = [np.array(v, dtype=np.uint64) for v in np.broadcast_arrays(*[np.asarray(v, dtype=np.uint64) for v in (*counters, k0, k1)])]
    c, (k0, k1) = c[:4], c[4:]
    low, half = np.uint64(0xFFFFFFFF), np.uint64(32)

    def mul(a, b):
        a = np.uint64(a)
        a0, a1, b0, b1 = a & low, a >> half, b & low, b >> half
        t = a1 * b0 + ((a0 * b0) >> half)
        hi = a1 * b1 + (t >> half) + (((t & low) + a0 * b1) >> half)
        return hi, a * b

    with np.errstate(over="ignore"):
        for _ in range(10):
            h0, l0 = mul(0xD2E7470EE14C6C93, c[0])
            h1, l1 = mul(0xCA5A826395121157, c[2])
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
            k0, k1 = k0 + np.uint64(0x9E3779B97F4A7C15), k1 + np.uint64(0xBB67AE8584CAA73B)
    return [(v >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 for v in c]


def exact_sweep(p, case, seed, sweeps):
    """Metropolis sweeps in double precision: every ratio from the bordered
    Pfaffian, every accepted change by the low-rank update of the inverses."""
    n, nl, r, h = case["n"], 2 * p.V, p.r, p.h2
    links = values(p, cold_links(case, n))
    cs, idx = constants(p), torch.from_numpy(link_indices(p)).to(device())
    ell = log_pfaffians(p, links[:1]).repeat(n, 1)
    W = []
    for k, (G, _, _) in enumerate(cs):
        D, tw = matrices(p, G, links[:1])
        inv = torch.linalg.inv(D + tw).expand(n, p.N, p.N)
        W.append((inv.real if k < p.K else inv).clone())
    logc, w = cplx([c[1] for c in cs]), cplx([c[2] for c in cs])
    real = torch.arange(p.P, device=device()) < p.K
    eye, obs = torch.eye(r, dtype=torch.complex128, device=device()), []
    for sweep in range(sweeps):
        accepted = torch.zeros(n, dtype=torch.float64, device=device())
        ctr = np.arange(nl, dtype=np.uint64)[:, None]
        u = philox((np.uint64(sweep), ctr, np.uint64(0), np.uint64(0)), np.uint64(seed), np.arange(n, dtype=np.uint64))
        u = [torch.from_numpy(v).to(device()) for v in u]
        for l in range(nl):
            old = links[:, l]
            if p.group_name == "Z2":
                new = -old
            elif p.group_name == "U1":
                new = old + WIDTH * (u[1][l] - 0.5)
                new = torch.where(new >= TWO_PI, new - TWO_PI, torch.where(new < 0, new + TWO_PI, new))
            else:
                d, z, ph = WIDTH * (u[1][l] - 0.5), 2.0 * u[2][l] - 1.0, TWO_PI * u[3][l]
                rho = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
                step = torch.stack([d.cos(), d.sin() * rho * ph.cos(), d.sin() * rho * ph.sin(), d.sin() * z], dim=-1)
                new = quat_mul(step, old)
                new = new / new.norm(dim=-1, keepdim=True)
            at = idx[l]
            delta = torch.stack([twisted(p, G, new) - twisted(p, G, old) for G, _, _ in cs], dim=1)
            wss = torch.stack([x[:, at[:, None], at[None, :]].to(torch.complex128) for x in W], dim=1)
            top = torch.cat([delta, -eye.expand_as(delta)], dim=-1)
            low = torch.cat([eye.expand_as(delta), wss], dim=-1)
            bord = torch.cat([top, low], dim=-2).reshape(n * p.P, 2 * r, 2 * r)
            la, ph = torch.zeros(n * p.P, dtype=torch.float64, device=device()), torch.ones(n * p.P, dtype=torch.complex128, device=device())
            eliminate(bord, 2 * r, la, ph)
            ratio = (la.exp() * ph).reshape(n, p.P)
            e = logc + ell
            e = torch.complex(e.real, torch.where(real, 0.0, e.imag))
            t = w * torch.exp(e - e.real.max(dim=1, keepdim=True).values)
            so, sn = t.real.sum(dim=1), (t * ratio).real.sum(dim=1)
            acc = (sn > 0) & (so > 0) & (u[0][l] < sn / so)
            accepted += acc
            Z = torch.linalg.solve(eye + delta @ wss, delta)
            lr = torch.complex(ratio.abs().log(), ratio.angle())
            grown = ell + torch.complex(lr.real, torch.where(real, 0.0, lr.imag))
            im = torch.where(grown.imag > math.pi, grown.imag - TWO_PI, torch.where(grown.imag <= -math.pi, grown.imag + TWO_PI, grown.imag))
            ell = torch.where(acc[:, None], torch.complex(grown.real, im), ell)
            links[:, l] = torch.where(acc.reshape((n,) + (1,) * (old.dim() - 1)), new, old)
            for k, x in enumerate(W):
                z = Z[:, k] * acc[:, None, None]
                z = z.real if k < p.K else z
                x.baddbmm_(x[:, :, at] @ z, x[:, at, :].clone(), alpha=-1)
        obs.append(torch.stack([plaquettes(p, links), terms(p, ell)[0], accepted / nl], dim=1))
    links = links.to(torch.int8) if p.group_name == "Z2" else links
    return {"obs": torch.stack(obs), "links": links, "ell": ell}


def net_loss(params, theta, origin, L):
    """Mean over the samples of -log q of the block links under the network."""
    s = torch.arange(L * L, device=theta.device)
    x, y = s % L, s // L
    inb = ((x - origin[:, :1]) % L < 4) & ((y - origin[:, 1:]) % L < 4)            # (b, V)
    right, up = y * L + (x + 1) % L, ((y + 1) % L) * L + x
    tx, ty = theta[:, 0::2], theta[:, 1::2]
    plaq = tx + ty[:, right] - tx[:, up] - ty
    out, free = ~inb, ~(inb | inb[:, right] | inb[:, up])
    X = torch.stack([tx.cos() * out, tx.sin() * out, ty.cos() * out, ty.sin() * out, plaq.cos() * free, plaq.sin() * free,
                     inb.double(), inb.double()], dim=1).reshape(-1, 8, L, L)
    at = 0
    for k, (ci, co) in enumerate(LAYERS):
        Wt, b = params[at:at + co * ci * 9].reshape(co, ci, 3, 3), params[at + co * ci * 9:at + co * ci * 9 + co]
        at += co * ci * 9 + co
        X = torch.nn.functional.conv2d(torch.nn.functional.pad(X, (1, 1, 1, 1), mode="circular"), Wt, b)
        X = torch.relu(X) if k < len(LAYERS) - 1 else X
    X = X.reshape(len(theta), 2, 3, L * L)
    total = 0.0
    for d, t in enumerate((tx, ty)):
        mu, rho = torch.atan2(X[:, d, 1], X[:, d, 0]), 0.95 * torch.sigmoid(X[:, d, 2])
        logf = torch.log1p(-rho * rho) - math.log(TWO_PI) - torch.log(1.0 + rho * rho - 2.0 * rho * torch.cos(t - mu))
        total = total - torch.where(inb, logf, torch.zeros_like(logf)).sum()
    return total / len(theta)


def exact_train(case, seed):
    L, batch = case["L"], case["batch"]
    theta = torch.from_numpy(net_data(case, seed)).to(device())
    x = torch.from_numpy(net_params(seed).astype(np.float64)).to(device())
    m, v, losses = torch.zeros_like(x), torch.zeros_like(x), []
    for step in range(case["steps"]):
        u = philox((np.uint64(step), np.arange(batch, dtype=np.uint64), np.uint64(13), np.uint64(0)), np.uint64(1), np.uint64(0x747261696E))
        cfg = np.minimum(case["n"] - 1, (u[0] * case["n"]).astype(np.int64))
        origin = np.stack([np.minimum(L - 1, (q * L).astype(np.int64)) for q in u[1:3]], axis=1)
        x.requires_grad_(True)
        loss = net_loss(x, theta[torch.from_numpy(cfg).to(device())], torch.from_numpy(origin).to(device()), L)
        (g,) = torch.autograd.grad(loss, x)
        losses.append(loss.item())
        with torch.no_grad():
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            x = x - 2e-3 * (m / (1 - 0.9 ** (step + 1))) / ((v / (1 - 0.999 ** (step + 1))).sqrt() + 1e-8)
    return {"losses": np.array(losses), "params": x.detach().cpu().numpy()}
