"""Performance cases of the Axilrod-Teller engine: what its users have it do.

Every case goes through the public Python entry points (`api.potential`,
`api.forces`, `api.Potential` with its backward pass, `api.farfield3`,
`api.Server`). Point sets are the ones of this repository's configurations:
uniform at unit density with minimum distance 0.5, the unit cube with minimum
distance 0.01, and isotropic Gaussian mixtures with minimum distance 0.05.

Results of the FP64 modes are kept in float64. The other modes (FP32 triple
arithmetic, tree, far-field) carry FP32 values in the entry point's float64
array, and a program that asks for them keeps them as float32 next to its other
single-precision features: `run` makes that conversion as such a program does.
"""
import math

import numpy as np
import torch

from paper_1105_2769_gb300 import api, inputs

DEV = "cuda"


def listed():
    return [
        # The smallest configured workload: 512 particles of the unit cube, FP64 reference sum.
        # Launches and latency count.
        {"name": "phi64_n512", "kind": "phi", "mode": "fp64", "set": "unit", "n": 512},
        # FP64 reference sum of a mid-sized ragged system (accuracy studies, force-field checks).
        {"name": "phi64_n3001", "kind": "phi", "mode": "fp64", "set": "uniform", "n": 3001},
        # One small system per call in FP32 bulk, as in a loop over molecules or serving requests.
        {"name": "phi32_n1000", "kind": "phi", "mode": "fp32", "set": "uniform", "n": 1000},
        # A clustered system of ordinary size with a ragged last tile.
        {"name": "phi32_mix_n5003", "kind": "phi", "mode": "fp32", "set": "mixture", "n": 5003},
        # The exhaustive FP32-bulk sum on a large uniform system (the benchmark's workload,
        # at a size whose pass stays below a second).
        {"name": "phi32_n20000", "kind": "phi", "mode": "fp32", "set": "uniform", "n": 20000},
        # Exhaustive forces, FP32 bulk: one step of molecular dynamics.
        {"name": "forces32_n8192", "kind": "forces", "mode": "fp32", "set": "uniform", "n": 8192},
        # Exhaustive forces in FP64: a small system, the reference for central differences.
        {"name": "forces64_n700", "kind": "forces", "mode": "fp64", "set": "uniform", "n": 700},
        # Forward and backward through autograd on float32 points: a training step that fits
        # positions or a model's output to potentials.
        {"name": "train32_n2500", "kind": "train", "mode": "fp32", "set": "uniform", "n": 2500},
        # Multi-tree potential at the configured eps = 1e-2, alpha = 0.05 on a clustered system.
        {"name": "tree_phi_n9000", "kind": "tree_phi", "eps": 1e-2, "alpha": 0.05,
         "set": "mixture", "n": 9000},
        # Multi-tree forces at the same setting: the serving workload's second request kind.
        {"name": "tree_forces_n3000", "kind": "tree_forces", "eps": 1e-2, "alpha": 0.05,
         "set": "mixture", "n": 3000},
        # Far-field expansion of order 4: 2^20 query points against two source clusters
        # of 4 096 points (the benchmark's workload).
        {"name": "farfield_p4_q1048576", "kind": "farfield", "p": 4, "nq": 1 << 20, "ns": 4096},
        # A burst of 12 requests on the batching server: sizes in [1 024, 4 096], 70 % tree
        # potentials and 30 % FP32 forces, half uniform and half clustered systems.
        {"name": "serve_burst12", "kind": "serve", "requests": 12, "nmin": 1024, "nmax": 4096},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["phi32", "phi32", "phi64", "forces32", "forces64", "train", "tree_phi",
                       "tree_forces", "farfield", "serve"])
    dist = rng.choice(["uniform", "mixture"])
    if kind == "phi32":
        return {"kind": "phi", "mode": "fp32", "set": dist, "n": _logint(rng, 60, 20000)}
    if kind == "phi64":
        return {"kind": "phi", "mode": "fp64", "set": rng.choice(["unit", "uniform", "mixture"]),
                "n": _logint(rng, 60, 3001)}
    if kind == "forces32":
        return {"kind": "forces", "mode": "fp32", "set": dist, "n": _logint(rng, 60, 8192)}
    if kind == "forces64":
        return {"kind": "forces", "mode": "fp64", "set": dist, "n": _logint(rng, 60, 1200)}
    if kind == "train":
        return {"kind": "train", "mode": "fp32", "set": dist, "n": _logint(rng, 60, 5000)}
    if kind == "tree_phi":
        return {"kind": "tree_phi", "eps": rng.choice([1e-2, 1e-1]), "alpha": 0.05, "set": dist,
                "n": _logint(rng, 500, 9000)}
    if kind == "tree_forces":
        return {"kind": "tree_forces", "eps": rng.choice([1e-2, 1e-1]), "alpha": 0.05, "set": dist,
                "n": _logint(rng, 300, 3000)}
    if kind == "farfield":
        return {"kind": "farfield", "p": rng.randint(0, 6), "nq": _logint(rng, 1000, 1 << 20),
                "ns": _logint(rng, 100, 8192)}
    return {"kind": "serve", "requests": rng.randint(4, 12), "nmin": 1024,
            "nmax": rng.randint(1500, 4096)}


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _points(which, n, seed):
    if which == "unit":  # density 512, so that larger sets keep the spacing
        return inputs.uniform_cube(n, max(1.0, (n / 512) ** (1 / 3)), 0.01, seed)
    if which == "uniform":
        return inputs.uniform_cube(n, n ** (1 / 3), 0.5, seed)
    # the serving workload's mixture: component volume density of the 2^20-point set
    comps = n // 16384 + 1
    side = 100.0 * (n / (1 << 20)) ** (1 / 3)
    return inputs.gaussian_mixture(n, comps, side, 0.5, 3.0, 0.05, seed)


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _clusters(nq, ns, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)

    def normal(n):
        return torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64) * 0.35

    c2 = torch.tensor([4.0, 0.3, -0.2], dtype=torch.float64, device=DEV)
    c3 = torch.tensor([0.5, 4.0, 1.6], dtype=torch.float64, device=DEV)
    return normal(nq), normal(ns) + c2, normal(ns) + c3


_kept = {}


def _server():
    """The process's request server: a program starts one and keeps it."""
    if "server" not in _kept:
        _kept["server"] = api.Server(0, hbm_budget_bytes=120 << 30, slots=8)
    return _kept["server"]


def _requests(case, seed):
    sizes = np.random.default_rng(case["requests"] * 10000 + case["nmax"])  # of the case alone
    reqs = []
    for q in range(case["requests"]):
        n = int(np.exp(sizes.uniform(np.log(case["nmin"]), np.log(case["nmax"]))))
        X = _points("uniform" if q % 2 else "mixture", n, seed * 100 + q)
        kind = "tree" if q % 10 < 7 else "forces"
        out = np.empty((n, 3) if kind == "forces" else n)
        reqs.append((kind, X, out))
    return reqs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "farfield":
        Xq, Y2, Y3 = _clusters(case["nq"], case["ns"], seed)
        return {"case": case, "Xq": Xq, "Y2": Y2, "Y3": Y3}
    if kind == "serve":
        return {"case": case, "server": _server(), "requests": _requests(case, seed)}
    X = _device(_points(case["set"], case["n"], seed))
    state = {"case": case, "X": X}
    if kind == "train":
        state["X"] = X.float().requires_grad_(True)
        state["g"] = _device(inputs.random_weights(case["n"], seed + 1))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "phi":
        phi = api.potential(state["X"], mode=case["mode"])
        return phi if case["mode"] == "fp64" else phi.float()
    if kind == "forces":
        F = api.forces(state["X"], mode=case["mode"])
        return F if case["mode"] == "fp64" else F.float()
    if kind == "train":
        phi = api.Potential.apply(state["X"], case["mode"])
        (grad,) = torch.autograd.grad(phi, state["X"], state["g"])
        return {"phi": phi.detach().float(), "grad": grad}
    if kind == "tree_phi":
        return api.potential(state["X"], mode="tree", eps=case["eps"], alpha=case["alpha"]).float()
    if kind == "tree_forces":
        return api.forces(state["X"], mode="tree", eps=case["eps"], alpha=case["alpha"]).float()
    if kind == "farfield":
        return api.farfield3(state["Xq"], state["Y2"], state["Y3"], case["p"]).float()
    srv = state["server"]
    tickets = []
    for what, X, out in state["requests"]:
        if what == "tree":
            tickets.append(srv.submit(X, mode="tree", eps=1e-2, alpha=0.05, out=out))
        else:
            tickets.append(srv.submit(X, kind="forces", mode="fp32", out=out))
    results = []
    for t in tickets:
        status, _, out = srv.poll(t)
        if status != 0:
            raise RuntimeError(f"request failed with status {status}")
        results.append(out.astype(np.float32))
    return results


# ---------------------------------------------------------------------------
# Work: each input read once, each output written once; 23 FLOPs per unordered
# triple for a potential (the direction-cosine form), 56 for the three members'
# gradients (the scatter form), and the expansion's coefficients per query.
# ---------------------------------------------------------------------------
def _triples(n):
    return n * (n - 1) * (n - 2) / 6.0


def _n_indices(p):
    return (p + 1) * (p + 2) * (p + 3) // 6


def work(case):
    kind = case["kind"]
    if kind == "farfield":
        p = case["p"]
        per = 0
        for d in range(p + 1):  # contractions of ten product terms
            per += 10 * (d + 1) * (d + 2) // 2 * (2 * _n_indices(p - d) + 2)
        per += 8 * 11 * _n_indices(p)  # Taylor coefficients of four powers at two centres
        return {"bytes": 24.0 * (case["nq"] + 2 * case["ns"]) + 4.0 * case["nq"],
                "flops": float(per * case["nq"])}
    if kind == "serve":
        n = math.sqrt(case["nmin"] * case["nmax"])
        r = case["requests"]
        return {"bytes": r * 40.0 * n, "flops": r * (0.7 * 23 + 0.3 * 56) * _triples(n)}
    n = case["n"]
    # At these sizes nearly all triples of a tree solve are base cases: counted as exhaustive.
    flops = {"phi": 23, "forces": 56, "train": 79, "tree_phi": 23, "tree_forces": 56}[kind]
    out = {"phi": 8, "forces": 24, "train": 20, "tree_phi": 4, "tree_forces": 12}[kind]
    return {"bytes": (24.0 + out) * n, "flops": flops * _triples(n)}


# ---------------------------------------------------------------------------
# The same values in 64 bits, by plain torch.
# ---------------------------------------------------------------------------
def _unit_pairs(X):
    d = X[None, :, :] - X[:, None, :]  # d[i, j] = x_j - x_i
    r = d.norm(dim=-1)
    r.fill_diagonal_(math.inf)
    return d / r[..., None], r


def _phi_exact(X):
    """Phi_i = sum_{j<k} (1 + 3 cos cos cos) / (r_ij r_ik r_jk)^3 from the definition."""
    n = X.shape[0]
    E, r = _unit_pairs(X)
    rho = r ** -3
    planes = [E[..., d].contiguous() for d in range(3)]
    phi = torch.zeros(n, dtype=torch.float64, device=X.device)
    for i in range(n):
        u = E[i]
        cos_i = u @ u.T
        # a_jk = e_ij . e_jk; cos_j = -a_jk, and cos_k = e_ik . e_jk = -a_kj
        a = u[:, 0:1] * planes[0] + u[:, 1:2] * planes[1] + u[:, 2:3] * planes[2]
        t = cos_i * a
        t *= a.T
        t.mul_(3.0).add_(1.0).mul_(rho)
        phi[i] = 0.5 * (rho[i] @ t @ rho[i])
    return phi


def _grad_exact(X, g=None):
    """sum over triples containing i of w grad_i phi, w = g_i + g_j + g_k (or 1)."""
    n = X.shape[0]
    E, r = _unit_pairs(X)
    rho = r ** -3
    inv = 1.0 / r
    planes = [E[..., d].contiguous() for d in range(3)]
    out = torch.zeros_like(X)
    for i in range(n):
        u = E[i]
        p1 = u @ u.T
        p2 = u[:, 0:1] * planes[0] + u[:, 1:2] * planes[1] + u[:, 2:3] * planes[2]
        p3 = -p2.T  # e_ik . e_jk
        R = rho[i][:, None] * rho[i][None, :] * rho
        if g is not None:
            R = R * (g[i] + g[:, None] + g[None, :])
        q = 5.0 * p1 * p2 * p3 - 1.0
        su = 3.0 * R * inv[i][:, None]
        sv = 3.0 * R * inv[i][None, :]
        c1 = su * q - sv * (p2 * p3)
        c2 = sv * q - su * (p2 * p3)
        c3 = su * (p1 * p3) + sv * (p1 * p2)
        c3 = torch.stack([(c3 * planes[d]).sum() for d in range(3)])
        out[i] = 0.5 * (c3 - c1.sum(1) @ u - c2.sum(0) @ u)
    return out


def _indices(p):
    return [(i, j, k - i - j) for k in range(p + 1) for i in range(k, -1, -1)
            for j in range(k - i, -1, -1)]


def _taylor(v, s2, p):
    """D^a (v.v)^(s2/2) / a! at the rows of v for every |a| <= p, in the order of _indices."""
    r2 = (v * v).sum(-1)
    ix = _indices(p)
    t = {(0, 0, 0): r2 ** (s2 / 2.0)}
    for a in ix[1:]:
        k = sum(a)
        one = torch.zeros_like(r2)
        two = torch.zeros_like(r2)
        for d in range(3):
            if a[d] >= 1:
                b = tuple(a[e] - (e == d) for e in range(3))
                one = one + v[..., d] * t[b]
            if a[d] >= 2:
                b = tuple(a[e] - 2 * (e == d) for e in range(3))
                two = two + t[b]
        t[a] = ((s2 - 2 * k + 2) * one + (s2 - k + 2) * two) / (k * r2)
    return torch.stack([t[a] for a in ix], dim=-1)


def _farfield_exact(Xq, Y2, Y3, p):
    """The p-th order Cartesian expansion of the product-term form, in 64 bits."""
    ix = _indices(p)
    pos = {a: q for q, a in enumerate(ix)}
    c2, c3 = Y2.mean(0), Y3.mean(0)
    fact = [math.factorial(k) for k in range(p + 1)]

    def moments(Y, c):
        d = Y - c
        return {a: float((d[:, 0] ** a[0] * d[:, 1] ** a[1] * d[:, 2] ** a[2]).sum())
                / (fact[a[0]] * fact[a[1]] * fact[a[2]]) for a in ix}

    M2, M3 = moments(Y2, c2), moments(Y3, c3)
    terms = {}
    for i, j, k, w in [(3, 0, 0, -1), (0, 3, 0, -1), (0, 0, 3, -1), (1, 1, 1, -2), (2, 1, 0, 1),
                       (2, 0, 1, 1), (1, 2, 0, 1), (0, 2, 1, 1), (1, 0, 2, 1), (0, 1, 2, 1)]:
        key = (2 * i - 5, 2 * j - 5, 2 * k - 5)
        terms[key] = terms.get(key, 0.0) + 0.375 * w
    terms[(-3, -3, -3)] += 1.0
    w23 = (c2 - c3)[None, :]
    D23 = {s: _taylor(w23, s, p)[0].tolist() for s in (1, -1, -3, -5)}
    tu = {s: _taylor(Xq - c2, s, p) for s in (1, -1, -3, -5)}
    tv = {s: _taylor(Xq - c3, s, p) for s in (1, -1, -3, -5)}

    def binom3(a, b):
        return math.comb(a[0], b[0]) * math.comb(a[1], b[1]) * math.comb(a[2], b[2])

    # S[s][a12, a13] = sum over a23 and its splits b + (a23 - b): x - c2 is displaced by
    # -(y2 - c2), c2 - c3 by (y2 - c2) - (y3 - c3).
    size = len(ix)
    S = {s: np.zeros((size, size)) for s in D23}
    for a12 in ix:
        for a13 in ix:
            left = p - sum(a12) - sum(a13)
            if left < 0:
                continue
            f12 = fact[a12[0]] * fact[a12[1]] * fact[a12[2]]
            f13 = fact[a13[0]] * fact[a13[1]] * fact[a13[2]]
            sign = -1.0 if (sum(a12) + sum(a13)) % 2 else 1.0
            for a23 in ix:
                if sum(a23) > left:
                    break
                f23 = fact[a23[0]] * fact[a23[1]] * fact[a23[2]]
                acc = 0.0
                for b0 in range(a23[0] + 1):
                    for b1 in range(a23[1] + 1):
                        for b2 in range(a23[2] + 1):
                            b = (b0, b1, b2)
                            c = tuple(a23[e] - b[e] for e in range(3))
                            m2 = tuple(a12[e] + b[e] for e in range(3))
                            m3 = tuple(a13[e] + c[e] for e in range(3))
                            acc += ((-1.0) ** sum(c) * binom3(m2, a12) * binom3(m3, a13)
                                    * M2[m2] * M3[m3])
                for s in D23:
                    # Taylor coefficient times a23! gives the derivative
                    S[s][pos[a12], pos[a13]] += sign * f12 * f13 * acc * D23[s][pos[a23]] * f23
    out = torch.zeros(Xq.shape[0], dtype=torch.float64, device=Xq.device)
    for (s12, s13, s23), w in terms.items():
        K = torch.from_numpy(S[s23]).to(Xq.device) * w
        out += ((tu[s12] @ K) * tv[s13]).sum(-1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "farfield":
        return _farfield_exact(*_clusters(case["nq"], case["ns"], seed), case["p"])
    if kind == "serve":
        out = []
        for what, X, _ in _requests(case, seed):
            X = _device(X)
            out.append(-_grad_exact(X) if what == "forces" else None)
        return out
    if case["n"] > {"forces": 4200, "train": 3000}.get(kind, 5200):
        return None  # takes too long in 64 bits
    if kind == "train":
        state = prepare(case, seed)
        X = state["X"].detach().double()
        return {"phi": _phi_exact(X), "grad": _grad_exact(X, state["g"])}
    X = _device(_points(case["set"], case["n"], seed))
    # A tree solve approximates the exhaustive result within eps: that is its exact value.
    return -_grad_exact(X) if kind in ("forces", "tree_forces") else _phi_exact(X)
