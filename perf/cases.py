"""Performance cases: what a program that uses this framework has it do.

Each case is one call sequence through the public entry points
(paper_0706_0747_gb300.mra) on inputs drawn from a seed: the adaptive apply of
a radial kernel at the orders, tolerances, precisions and screens in use, the
batched apply, the ground-state iteration, the two-dimensional variant,
Algorithm 1, the two-scale transforms and the learned schedule's network.
``exact`` restates each of them in 64 bits with plain torch, from the same
input trees and operator tables.
"""
import ctypes
import math

import numpy as np
import torch

from paper_0706_0747_gb300 import mra, workloads as W

TC = ("tc", "tc_ladder")
EPS_OF = {4: 1e-4, 5: 1e-4, 6: 1e-5, 7: 1e-5, 8: 1e-6, 10: 1e-6}


# ---------------------------------------------------------------- the cases
def _apply(name, k, gaussians, lo, hi, precision, screen="static", mu=0.0, levels=7, uniform=-1):
    return {"name": name, "kind": "apply", "k": k, "eps": EPS_OF[k], "mu": mu, "levels": levels, "uniform": uniform,
            "gaussians": gaussians, "log_lo": lo, "log_hi": hi, "precision": precision, "screen": screen}


def listed():
    return [
        # the smallest call: a uniform level-3 tree (585 nodes) at low order, where launches and
        # host latency count -- a coarse potential inside someone else's inner loop
        _apply("uniform_k4_tc", 4, 4, 2.0, 3.0, "tc", levels=3, uniform=3),
        # bound-state Helmholtz kernel on a few hundred nodes (one step of an eigenvalue iteration)
        _apply("helmholtz_k8_tc", 8, 5, 1.0, 2.5, "tc", mu=1.5, levels=8),
        # the benchmark's workload with the default (static) screen: compress, apply, assemble
        _apply("poisson_k8_tc", 8, 64, 2.0, 5.0, "tc"),
        # the same with the exact per-pair screen
        _apply("poisson_k8_tc_pair", 8, 64, 2.0, 5.0, "tc", screen="pair"),
        # the reference precision, on resolved densities
        _apply("poisson_k8_fp64", 8, 16, 2.0, 3.5, "fp64"),
        # an odd order in single precision
        _apply("poisson_k5_fp32", 5, 9, 1.0, 3.5, "fp32"),
        # many right-hand sides: screen and apply of a batch, one output tree per input
        {"name": "batch_k6_tc", "kind": "batch", "k": 6, "eps": 1e-5, "mu": 0.0, "levels": 7, "trees": 32,
         "gaussians": 16, "log_lo": 1.0, "log_hi": 4.0, "precision": "tc", "screen": "static"},
        # one step of the hydrogen ground-state iteration with a kept operator
        {"name": "hydrogen_k8_tc", "kind": "kalos", "k": 8, "eps": 1e-6, "levels": 12, "init": 3,
         "precision": "tc", "screen": "static"},
        # the two-dimensional variant: compress, apply, assemble and truncate
        {"name": "square_k8_fp64", "kind": "apply2", "k": 8, "eps": 1e-6, "mu": 0.0, "alpha": 0.5, "levels": 12,
         "gaussians": 64, "log_lo": 2.5, "log_hi": 5.0},
        # Algorithm 1 on a new density
        {"name": "build_k8", "kind": "build", "k": 8, "eps": 1e-6, "levels": 7, "gaussians": 32, "log_lo": 2.0,
         "log_hi": 4.5},
        # decomposition with stored wavelet blocks and back
        {"name": "roundtrip_k8", "kind": "roundtrip", "k": 8, "eps": 1e-6, "levels": 7, "gaussians": 64,
         "log_lo": 2.0, "log_hi": 5.0},
        # a training batch of the learned schedule: loss, gradients, and the predictions
        {"name": "schedule_4096", "kind": "schedule", "rows": 4096},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "batch", "kalos", "apply2", "build", "roundtrip",
                       "schedule"])
    lo = rng.uniform(1.0, 2.5)
    if kind == "apply":
        precision = rng.choice(["tc", "tc", "tc", "tc_ladder", "fp32", "fp64"])
        k = rng.choice([4, 5, 6, 7, 8] if precision in TC else [4, 5, 6, 7, 8, 10])
        most = 48 if precision in TC else (12 if k <= 8 else 3)
        c = _apply("", k, _logint(rng, 1, most), lo, lo + rng.uniform(0.5, 2.0), precision,
                   screen=rng.choice(["static", "static", "pair"]), mu=rng.choice([0.0, 0.0, 1.5, 4.0]),
                   levels=rng.choice([4, 5, 6, 7, 8]))
    elif kind == "batch":
        k = rng.choice([4, 6, 8])
        c = {"kind": "batch", "k": k, "eps": EPS_OF[k], "mu": rng.choice([0.0, 1.5]), "levels": rng.choice([5, 6, 7]),
             "trees": _logint(rng, 2, 24), "gaussians": _logint(rng, 1, 12), "log_lo": lo, "log_hi": lo + 1.0,
             "precision": "tc", "screen": rng.choice(["static", "pair"])}
    elif kind == "kalos":
        k = rng.choice([5, 6, 8])
        c = {"kind": "kalos", "k": k, "eps": EPS_OF[k], "levels": rng.randint(6, 12), "init": rng.choice([2, 3]),
             "precision": rng.choice(["tc", "tc", "fp64"]), "screen": rng.choice(["static", "pair"])}
    elif kind == "apply2":
        k = rng.choice([5, 6, 8])
        c = {"kind": "apply2", "k": k, "eps": EPS_OF[k], "mu": rng.choice([0.0, 0.0, 2.0]),
             "alpha": rng.choice([0.5, 0.75]), "levels": rng.randint(6, 12), "gaussians": _logint(rng, 2, 64),
             "log_lo": lo + 0.5, "log_hi": lo + 2.0}
    elif kind in ("build", "roundtrip"):
        k = rng.choice([4, 5, 6, 8, 10])
        c = {"kind": kind, "k": k, "eps": EPS_OF[k], "levels": rng.choice([5, 6, 7]),
             "gaussians": _logint(rng, 1, 32 if k <= 8 else 4), "log_lo": lo, "log_hi": lo + 2.0}
    else:
        c = {"kind": "schedule", "rows": _logint(rng, 100, 12000)}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs
def _density(case, rng, dim=3, instance=0):
    """Unit-mass Gaussians, log10 exponents U[log_lo, log_hi], centres U[0.15, 0.85]^dim: the mesh
    they need belongs to the case.  The seed's own generator turns them by one of the cube's
    symmetries and weighs them, so that inputs differ while their trees keep their size."""
    base = np.random.default_rng([case["k"], case["gaussians"], round(1000 * case["log_lo"]), instance])
    expo = 10.0 ** base.uniform(case["log_lo"], case["log_hi"], case["gaussians"])
    cen = base.uniform(0.15, 0.85, (case["gaussians"], dim))[:, rng.permutation(dim)]
    cen = np.where(rng.random(dim) < 0.5, cen, 1.0 - cen)
    d = W.unit_mass(expo, cen) if dim == 3 else W.unit_mass2(expo, cen)
    d.coef = d.coef * math.exp(rng.uniform(-1.0, 1.0))
    return d


def _tree(case, rng, instance=0):
    d = _density(case, rng, instance=instance)
    t, _ = mra.build_tree(d, case["k"], case["eps"], case["levels"], uniform_level=case.get("uniform", -1),
                          init_level=2)
    return t


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind in ("apply", "batch"):
        s["op"] = mra.make_operator(case["mu"], 1.0, case["eps"], case["k"], case["levels"])
        s["trees"] = [_tree(case, rng, b) for b in range(case.get("trees", 1))]
    elif kind == "apply2":
        s["op"] = mra.make_operator2(case["mu"], case["alpha"], case["eps"], case["k"], case["levels"])
        d = _density(case, rng, dim=2)
        s["tree"], _ = mra.build_tree2(d, case["k"], case["eps"], case["levels"], init_level=2)
    elif kind == "kalos":
        # one step from exp(-zeta r) builds the operator; the measured step re-weights it
        h = W.Hydrogen("hydrogen", 32.0, (0.5, 0.5, 0.5), 0.7, rng.uniform(0.76, 0.82), case["k"], case["eps"],
                       case["levels"], case["init"])
        s["length"] = h.L
        s["potential"] = mra.Potential(charges=[-1.0 / h.L], positions=[h.u0])
        s["cache"] = mra.OpCache()
        phi, _ = mra.build_tree(h.start_density(), h.k, h.eps, h.max_level, init_level=h.init_level)
        mra.tree_scale(phi, 1.0 / math.sqrt(mra.tree_dot(phi, phi) * h.L ** 3))
        s["phi"], _ = mra.kalos_step(phi, s["potential"], h.L, h.mu0, h.eps, h.max_level,
                                     precision=case["precision"], screen=case["screen"], op_cache=s["cache"])
        s["mu"] = rng.uniform(0.85, 0.95)
    elif kind == "build":
        s["density"] = _density(case, rng)
    elif kind == "roundtrip":
        s["tree"] = _tree(case, rng)
    else:
        s["net"] = mra.mlp_create(seed=seed)
        # the 16 inputs of a box: scaled logarithms and fractions; the targets: a flag and two fractions
        n = case["rows"]
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        s["x"] = torch.rand((n, 16), generator=g, device="cuda") * 2 - 0.5
        y = torch.rand((n, 4, 3), generator=g, device="cuda")
        y[..., 0] = (y[..., 0] < 0.3).float()
        y[..., 1:] *= 1 - y[..., :1]
        s["target"] = y.reshape(n, 12).contiguous()
    return s


class _View:
    """A tree's device array as torch sees it; holds the tree."""

    def __init__(self, tree, ptr, shape, typestr):
        self.tree = tree
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (ptr, False), "version": 3}


def _arrays(tree):
    """(blocks, leaf flags) of a tree in place."""
    inf = tree.info()
    b, leaf = tree.device_arrays()
    k = inf.k
    return (torch.as_tensor(_View(tree, b, (inf.n_nodes, k, k, k), "<f8"), device="cuda"),
            torch.as_tensor(_View(tree, leaf, (inf.n_nodes,), "<i4"), device="cuda"))


def _result(tree, precision):
    """A result's blocks; a program that chose 32-bit arithmetic (in registers or in the tensor
    cores' accumulators) takes them on in float32."""
    b = _arrays(tree)[0]
    return b if precision == "fp64" else b.float()


# ---------------------------------------------------------------- one pass
def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "apply":
        tree = s["trees"][0]
        mra.compress(tree, norms=False)
        g, _ = mra.apply_ns(s["op"], tree, precision=case["precision"], screen=case["screen"])
        mra.reconstruct(g, mode="assemble")
        return _result(g, case["precision"])
    if kind == "batch":
        for t in s["trees"]:
            mra.compress(t, norms=False)
        plan = mra.plan_create(s["op"], s["trees"], precision=case["precision"], use_graph=False,
                               screen=case["screen"])
        plan.execute()
        out = [_result(plan.output(b), case["precision"]) for b in range(len(s["trees"]))]
        plan.free()
        return out
    if kind == "apply2":
        mra.compress2(s["tree"])
        g, _ = mra.apply_ns2(s["op"], s["tree"])
        mra.reconstruct2(g, truncate=True, eps=case["eps"])
        coords, leaf, blocks, _ = g.export()
        return [coords, leaf, blocks]
    if kind == "kalos":
        phi, info = mra.kalos_step(s["phi"], s["potential"], s["length"], s["mu"], case["eps"], case["levels"],
                                   precision=case["precision"], screen=case["screen"], op_cache=s["cache"])
        r = np.array([info["energy"], info["mu_next"], info["norm_new"]])
        return [_result(phi, case["precision"]), r if case["precision"] == "fp64" else r.astype(np.float32)]
    if kind == "build":
        tree, _ = mra.build_tree(s["density"], case["k"], case["eps"], case["levels"], init_level=2)
        return list(_arrays(tree))
    if kind == "roundtrip":
        mra.compress(s["tree"], store_d=True)
        mra.reconstruct(s["tree"], mode="inverse")
        return _arrays(s["tree"])[0]
    loss, grad = s["net"].loss_grad(s["x"], s["target"])
    y = torch.empty((case["rows"], 12), device="cuda")
    s["net"].forward(s["x"], y)
    return [np.float32(loss), grad, y]


# ---------------------------------------------------------------- what a pass cannot do without
_counted = {}


def work(case):
    """Blocks in and out once; of the arithmetic the innermost contraction of every kept item
    (2 k^4 in three dimensions, 2 k^3 in two), counted on one input of the case."""
    key = tuple(sorted((a, b) for a, b in case.items() if a != "name"))
    if key not in _counted:
        _counted[key] = _work(case)
    return dict(_counted[key])


def _work(case):
    kind = case["kind"]
    if kind == "schedule":
        p = 16 * 128 + 2 * 128 * 128 + 128 * 12
        return {"bytes": 4.0 * (case["rows"] * (16 + 12 + 12) + 2 * p), "flops": 2.0 * p * case["rows"] * 4}
    s, k = prepare(case, 1), case["k"]
    if kind in ("apply", "batch"):
        items = nodes = 0
        for t in s["trees"]:
            mra.compress(t, norms=False)
            items += mra.apply_ns(s["op"], t, precision="fp32", screen=case["screen"])[1]["n_items"]
            nodes += t.n
        return {"bytes": 2.0 * nodes * k ** 3 * 8, "flops": 2.0 * k ** 4 * items}
    if kind == "apply2":
        mra.compress2(s["tree"])
        items = mra.apply_ns2(s["op"], s["tree"])[1]["n_items"]
        return {"bytes": 2.0 * s["tree"].n * k * k * 8, "flops": 2.0 * k ** 3 * items}
    if kind == "kalos":
        items = mra.kalos_step(s["phi"], s["potential"], s["length"], s["mu"], case["eps"], case["levels"],
                               precision="fp32", op_cache=s["cache"])[1]["n_items"]
        return {"bytes": 2.0 * s["phi"].n * k ** 3 * 8, "flops": 2.0 * k ** 4 * items}
    n = s["tree"].n if kind == "roundtrip" else run(s)[0].shape[0]
    if kind == "build":  # every box's values, and those of its children's grids
        return {"bytes": 1.0 * n * k ** 3 * 8, "flops": 9.0 * n * k ** 3 * 2 * case["gaussians"]}
    return {"bytes": 3.0 * n * k ** 3 * 8, "flops": n / 8 * 2 * 3 * 2 * (2.0 * k) ** 4}


# ---------------------------------------------------------------- 64 bits, plain torch
F64 = torch.float64


def _phi(k, u):
    """phi_i(u) = sqrt(2i + 1) P_i(2u - 1), rows i."""
    return np.stack([math.sqrt(2 * i + 1) * np.polynomial.legendre.legval(2 * u - 1, np.eye(k)[i]) for i in range(k)])


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (x + 1) / 2, w / 2


def _filters(k):
    """H^(p)[i][a] = (1/sqrt 2) int phi_i((u + p)/2) phi_a(u) du."""
    u, w = _gauss(k + 1)
    h = [(_phi(k, (u + p) / 2) * w) @ _phi(k, u).T / math.sqrt(2.0) for p in range(2)]
    return torch.tensor(np.stack(h), device="cuda")


def _along(x, mat, axis):
    """mat (out x in) along a trailing axis of the blocks x (n, k, ..., k)."""
    return torch.movedim(torch.tensordot(x, mat, dims=([axis], [1])), -1, axis)


def _spread(v, dim):
    out = torch.zeros_like(v)
    for b in range(13):
        out |= ((v >> b) & 1) << (dim * b)
    return out


def _key(box):
    dim = box.shape[1]
    k = torch.zeros(box.shape[0], dtype=torch.int64, device=box.device)
    for d in range(dim):
        k |= _spread(box[:, d], dim) << (dim - 1 - d)
    return k


class _Tree64:
    """A tree as tensors, nodes by level then key, and its redundant blocks."""

    def __init__(self, coords, leaf, blocks):
        c = torch.as_tensor(coords, device="cuda").long()
        self.level, self.box = c[:, 0], c[:, 1:]
        self.leaf = torch.as_tensor(leaf, device="cuda").bool()
        self.s = torch.as_tensor(blocks, device="cuda").clone()
        self.dim, self.k, self.n = self.box.shape[1], self.s.shape[1], len(c)
        self.H = _filters(self.k)
        self.nlev = int(self.level.max()) + 1
        self.key = _key(self.box)
        self.rows = [torch.nonzero(self.level == j)[:, 0] for j in range(self.nlev)]
        # an internal node's children are the next level's groups of 2^dim, in order
        g = 2 ** self.dim
        self.first = torch.full((self.n,), -1, dtype=torch.int64, device="cuda")
        for j in range(self.nlev - 1):
            inner = self.rows[j][~self.leaf[self.rows[j]]]
            self.first[inner] = self.rows[j + 1][0] + g * torch.arange(len(inner), device="cuda")

    def inner(self, j):
        return self.rows[j][~self.leaf[self.rows[j]]]

    def up(self, x, octant):
        """x (n, k..k) refined to the children `octant` (n,): d = 0."""
        out = torch.empty_like(x)
        for o in range(2 ** self.dim):
            m = octant == o
            if m.any():
                y = x[m]
                for d in range(self.dim):
                    y = _along(y, self.H[(o >> (self.dim - 1 - d)) & 1].T, d + 1)
                out[m] = y
        return out

    def parents_of_children(self, j):
        acc = 0
        rows = self.inner(j)
        for o in range(2 ** self.dim):
            y = self.s[self.first[rows] + o]
            for d in range(self.dim):
                y = _along(y, self.H[(o >> (self.dim - 1 - d)) & 1], d + 1)
            acc = acc + y
        return acc

    def compress(self):
        for j in range(self.nlev - 2, -1, -1):
            self.s[self.inner(j)] = self.parents_of_children(j)

    def assemble(self):
        """Children add their parent's refinement, from the root down."""
        for j in range(self.nlev - 1):
            rows = self.inner(j)
            for o in range(2 ** self.dim):
                self.s[self.first[rows] + o] += self.up(self.s[rows], torch.full_like(rows, o))

    def truncate(self, eps):
        """Merge leaf siblings whose parent's wavelet norm is small; the kept nodes."""
        dims = list(range(1, self.dim + 1))
        thr = eps * self.s[self.leaf].square().sum().sqrt() / math.sqrt(self.n)
        alive = torch.ones(self.n, dtype=torch.bool, device="cuda")
        leaf = self.leaf.clone()
        for j in range(self.nlev - 2, -1, -1):
            rows = self.inner(j)
            if not len(rows):
                continue
            d2 = 0
            small = torch.ones(len(rows), dtype=torch.bool, device="cuda")
            for o in range(2 ** self.dim):
                c = self.first[rows] + o
                d2 = d2 + (self.s[c] - self.up(self.s[rows], torch.full_like(rows, o))).square().sum(dims)
                small &= leaf[c]
            small &= d2.sqrt() < thr
            leaf[rows[small]] = True
            for o in range(2 ** self.dim):
                alive[self.first[rows[small]] + o] = False
        return alive, leaf

    def blocks_at(self, j, key):
        """Blocks of the boxes `key` (unique) of level j: nodes, or refined from the covering leaf."""
        have = self.key[self.rows[j]]
        at = torch.searchsorted(have, key).clamp(max=len(have) - 1)
        found = have[at] == key
        out = torch.empty((len(key),) + tuple(self.s.shape[1:]), dtype=F64, device="cuda")
        out[found] = self.s[self.rows[j][at[found]]]
        if not found.all():
            miss = key[~found]
            par, back = torch.unique(miss >> self.dim, return_inverse=True)
            out[~found] = self.up(self.blocks_at(j - 1, par)[back], miss & (2 ** self.dim - 1))
        return out


def _term_sum(x, wt, F):
    """sum_m wt[m, n] (F[0][m] x ... x F[d-1][m]) x[n]: x (n, k..k), F[d] (M, k, k)."""
    M, k, dim = wt.shape[0], x.shape[1], x.dim() - 1
    out = torch.zeros_like(x)
    step = max(1, int(4e7 // (M * k ** dim)))
    for a in range(0, len(x), step):
        y, w = x[a:a + step], wt[:, a:a + step]
        n = len(y)
        if dim == 3:
            z = torch.matmul(y.reshape(1, n * k * k, k), F[2].transpose(1, 2))             # (M, n k k, k)
            z = torch.matmul(F[1].reshape(M, 1, k, k), z.reshape(M, n * k, k, k))          # (M, n k, k, k)
            z = z.reshape(M, n, k, k * k) * w[:, :, None, None]
        else:
            z = torch.matmul(y.reshape(1, n * k, k), F[1].transpose(1, 2)).reshape(M, n, k, k) * w[:, :, None, None]
        z = z.permute(1, 0, 2, 3).reshape(n, M * k, -1)
        out[a:a + step] = torch.matmul(F[0].permute(1, 0, 2).reshape(k, M * k), z).reshape(y.shape)
    return out


def _apply64(op, T, eps, screen):
    """Algorithm 3 on the redundant tree T with the operator tables op: per-scale outputs."""
    dim, k, nlev = T.dim, T.k, T.nlev
    w, F, nF, est = (torch.as_tensor(op[q], device="cuda") for q in ("w", "F", "nF", "est"))
    M = len(w)
    root = T.s[T.rows[0]]
    F0 = [F[0, :, 3]] * dim
    sigma = _term_sum(root, w[:, None].clone(), F0).square().sum().sqrt()
    fnorm = T.s[T.leaf].square().sum().sqrt()
    eta = eps * sigma / fnorm
    Jm = torch.zeros(M, dtype=torch.int64, device="cuda")
    for j in range(1, nlev):
        Jm[w * est[j] > eta / M] = j
    budget = float(eta) / (2.0 * 6 ** dim)
    core, off = nF[:, :, 2:5].amax(2), nF[:, :, [0, 1, 5, 6]].amax(2)
    eta_blk = eps * sigma / math.sqrt(T.n * 6.0 ** dim * M)
    out = torch.zeros_like(T.s)
    for j in range(nlev):
        rows, N = T.rows[j], 1 << j
        act = (Jm >= j).cpu().numpy()
        cand = np.nonzero(act)[0]
        ranges = []
        for S in range(dim + 1):
            e = (w * core[j] ** S * off[j] ** (dim - S)).cpu().numpy()[cand]
            lo, hi, acc = 0, len(cand) - 1, 0.0
            while lo < len(cand) and acc + e[lo] <= budget:
                acc, lo = acc + e[lo], lo + 1
            acc = 0.0
            while hi >= lo and acc + e[hi] <= budget:
                acc, hi = acc + e[hi], hi - 1
            ranges.append(np.arange(M)[(np.arange(M) >= cand[lo]) & (np.arange(M) <= cand[hi]) & act]
                          if hi >= lo and len(cand) else np.zeros(0, int))
        # every pair of the level: per translation, the outputs and the keys of their inputs
        pairs, keys = [], []
        for t in np.ndindex(*([7] * dim)):
            t = [v - 3 for v in t]
            S = sum(abs(v) <= 1 for v in t)
            if not len(ranges[S]):
                continue
            b = T.box[rows] - torch.tensor(t, device="cuda")
            odd = T.box[rows] & 1
            ok = ((b >= 0) & (b < N)).all(1)
            for d in range(dim):
                ok &= (t[d] >= -3 + odd[:, d]) & (t[d] <= 2 + odd[:, d])
            if S == dim:  # internal nodes leave the core of terms that go on to finer scales
                here = bool((Jm[torch.as_tensor(ranges[S], device="cuda")] == j).any())
                ok &= T.leaf[rows] | here
            if ok.any():
                pairs.append((t, S, rows[ok]))
                keys.append(_key(b[ok]))
        if not pairs:
            continue
        uniq, back = torch.unique(torch.cat(keys), return_inverse=True)
        X = T.blocks_at(j, uniq)
        norms = X.reshape(len(X), -1).square().sum(1).sqrt()
        at = 0
        for (t, S, a), kk in zip(pairs, keys):
            b = back[at:at + len(kk)]
            at += len(kk)
            m = torch.as_tensor(ranges[S], device="cuda")
            keep = torch.ones((len(m), len(a)), dtype=torch.bool, device="cuda")
            if S == dim:
                keep &= T.leaf[a][None] | (Jm[m] == j)[:, None]
            if screen == "pair":
                p = w[m]
                for d in range(dim):
                    p = p * nF[j, m, t[d] + 3]
                good = keep & (p[:, None] * norms[b][None] > eta_blk)
                first = torch.cumsum(good, 0) > 0
                last = torch.flip(torch.cumsum(torch.flip(good, [0]), 0), [0]) > 0
                keep &= first & last
            use = keep.any(1)
            if not use.any():
                continue
            wt = (w[m][:, None] * keep)[use]
            out[a] += _term_sum(X[b], wt, [F[j, m[use], t[d] + 3] for d in range(dim)])
    T.s = out


def _values(x, Phi):
    for d in range(3):
        x = _along(x, Phi, d + 1)
    return x


def _times(T, s, potential, scale):
    """scale V f on the leaves, projected by each box's k-point rule."""
    u, wq = _gauss(T.k)
    Phi = torch.tensor(_phi(T.k, u).T.copy(), device="cuda")
    u, wq = torch.tensor(u, device="cuda"), torch.tensor(wq, device="cuda")
    rows = torch.nonzero(T.leaf)[:, 0]
    x = [(T.box[rows, d, None] + u) / 2.0 ** T.level[rows, None] for d in range(3)]
    v = 0
    for q, r in zip(potential.charges, potential.positions.reshape(-1, 3)):
        d2 = ((x[0] - r[0]) ** 2)[:, :, None, None] + ((x[1] - r[1]) ** 2)[:, None, :, None] + \
            ((x[2] - r[2]) ** 2)[:, None, None, :]
        v = v + q / d2.sqrt()
    f = _values(s[rows], Phi) * v * scale * wq[:, None, None] * wq[:, None] * wq
    out = torch.zeros_like(s)
    out[rows] = _values(f, Phi.T)
    return out


def _build64(case, d):
    """Algorithm 1: blocks and leaf flags, level by level."""
    k, dev = case["k"], "cuda"
    c, a, cen = (torch.tensor(np.asarray(v), device=dev) for v in (d.coef, d.expo, d.centers))
    u, wq = _gauss(k)
    P = torch.tensor(_phi(k, u) * wq, device=dev)
    Q = [torch.tensor(_phi(k, (u + p) / 2).T.copy(), device=dev) for p in range(2)]
    u = torch.tensor(u, device=dev)

    def values(box, j):
        out = []
        for bx in box.split(1024):
            e = [torch.exp(-a[None, :, None] * ((bx[:, None, i, None] + u) / 2.0 ** j - cen[None, :, i, None]) ** 2)
                 for i in range(3)]
            yz = (e[1][:, :, :, None] * e[2][:, :, None, :]).reshape(len(bx), len(a), k * k)
            out.append(torch.bmm((c[None, :, None] * e[0]).transpose(1, 2), yz).reshape(-1, k, k, k))
        return torch.cat(out)

    r2 = (cen[:, None] - cen[None]).square().sum(2)
    tol = case["eps"] * (c[None] * torch.exp(-a[None] * r2)).sum(1).abs().max()
    box, blocks, leaves = torch.zeros((1, 3), dtype=torch.int64, device=dev), [], []
    for j in range(case["levels"] + 1):
        s = values(box, j)
        for ax in range(3):
            s = _along(s, P, ax + 1)
        s = s * 2.0 ** (-1.5 * j)
        octs = [torch.tensor([o >> 2, (o >> 1) & 1, o & 1], device=dev) for o in range(8)]
        if j < 2:
            split = torch.ones(len(box), dtype=torch.bool, device=dev)
        else:
            err = torch.zeros(len(box), dtype=F64, device=dev)
            for o in range(8):
                y = s
                for ax in range(3):
                    y = _along(y, Q[(o >> (2 - ax)) & 1], ax + 1)
                e = (values(2 * box + octs[o], j + 1) - y * 2.0 ** (1.5 * j)).abs().amax((1, 2, 3))
                err = torch.maximum(err, e)
            split = err > tol
        if j == case["levels"]:
            split[:] = False
        blocks.append(s)
        leaves.append(~split)
        if not split.any():
            break
        box = torch.stack([2 * box[split] + o for o in octs], 1).reshape(-1, 3)
    return [torch.cat(blocks), torch.cat(leaves).int()]


def _net64(s):
    """Loss, gradients and predictions: FP16 weights and activations, the rest in 64 bits."""
    p = torch.tensor(s["net"].get_params(), device="cuda")
    half = lambda t: t.half().double()  # noqa: E731
    Ws, at = [], 0
    for i, o in ((16, 128), (128, 128), (128, 128), (128, 12)):
        Ws.append((half(p[at:at + i * o].reshape(o, i)), p[at + i * o:at + i * o + o].double()))
        at += i * o + o
    hs = [s["x"].double()]
    for q, (w, b) in enumerate(Ws):
        z = hs[-1] @ w.T + b
        hs.append(half(z.float().clamp(min=0)) if q < 3 else z)
    y, t = hs[-1].reshape(-1, 4, 3), s["target"].double().reshape(-1, 4, 3)
    e, E, n = y[..., 0], t[..., 0], len(y)
    diff = y[..., 1:] - t[..., 1:]
    loss = (torch.nn.functional.softplus(e) - E * e + (1 - E) * diff.square().sum(2)).sum() / n
    d = torch.cat([(torch.sigmoid(e) - E)[..., None], 2 * (1 - E)[..., None] * diff], 2).reshape(n, 12) / n
    grads = []
    for q in range(3, -1, -1):
        w, b = Ws[q]
        grads = [torch.cat([(d.T @ hs[q]).reshape(-1), d.sum(0)])] + grads
        if q:
            d = (d @ w) * (hs[q] > 0)
    return [loss.cpu().numpy(), torch.cat(grads), hs[-1]]


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "schedule":
        return _net64(s)
    if kind == "build":
        return _build64(case, s["density"])
    if kind in ("apply", "batch"):
        op = s["op"].export()
        out = []
        for t in s["trees"]:
            T = _Tree64(*t.export()[:3])
            T.compress()
            _apply64(op, T, case["eps"], case["screen"])
            if kind == "apply":
                T.assemble()
                T.compress()
            out.append(T.s)
        return out[0] if kind == "apply" else out
    if kind == "apply2":
        T = _Tree64(*s["tree"].export()[:3])
        T.compress()
        _apply64(s["op"].export(), T, case["eps"], "static")
        T.assemble()
        T.compress()
        alive, leaf = T.truncate(case["eps"])
        coords = torch.cat([T.level[:, None], T.box], 1)
        return [coords[alive].int(), leaf[alive].int(), T.s[alive]]
    if kind == "roundtrip":
        T = _Tree64(*s["tree"].export()[:3])
        T.compress()
        return T.s
    # the ground-state step: the operator's tables as they are for this mu
    run(s)
    op = mra.Operator(ctypes.c_void_p(s["cache"].h.value))
    tables = op.export()
    op.h = None  # the cache owns it
    T = _Tree64(*s["phi"].export()[:3])
    P = _times(T, T.s, s["potential"], 1.0)
    T.s = P.clone()
    T.compress()
    _apply64(tables, T, case["eps"], case["screen"])
    T.assemble()
    L, mu = s["length"], s["mu"]
    new = T.s * (-2.0 * L * L)
    dot = lambda x, y: float((x[T.leaf] * y[T.leaf]).sum())  # noqa: E731
    nn = dot(new, new)
    e = (-dot(P, new) - 0.5 * mu * mu * nn + dot(_times(T, new, s["potential"], 1.0), new)) / nn
    norm = math.sqrt(nn * L ** 3)
    return [new / norm, np.array([e, math.sqrt(-2 * e) if e < 0 else mu, norm])]
