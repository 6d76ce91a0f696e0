"""What this library is used for, as cases that can be timed and checked.

Every case is one pass through the public binding (``paper_2503_13075_gb300.binding``): a
constraint solve of one time step, a learned warm start, or a gradient of the warm-start
network.  The topologies are the repository's own synthetic workloads (chains, tree-shaped
molecules, one protein-like system); a case fixes the topology, the seed draws the state of
the time step (orientations and places of the molecules, the unconstrained positions).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2503_13075_gb300 import binding as B
from paper_2503_13075_gb300 import workloads as wl

TOL = 1e-12  # relative violation every solve reaches (the binding's default)


def _solve(name, kind, **kw):
    c = {"name": name, "kind": kind, "n_mol": 1, "lo": 0, "hi": 0, "topology": 1, "precision": "mixed",
         "start": "diag", "overlap": 0, "host": False, "xoh": False}
    c.update(kw)
    return c


def listed():
    return [
        # one unbranched molecule of 64 atoms: the smallest call a time-stepping loop makes, where
        # launches and the chain of dependent steps are everything; in the mixed precision most
        # callers take, and in plain float64 from the paper's zero start
        _solve("chain64_mixed", "chain", lo=64, hi=64),
        _solve("chain64_fp64", "chain", lo=64, hi=64, precision="fp64", start="zero"),
        # a box of lipid-sized molecules of uneven size, every bond constrained: the ordinary
        # time step of a molecular simulation, mixed and in plain float64
        _solve("trees4096_mixed", "trees", n_mol=4096, lo=20, hi=200),
        _solve("trees4096_fp64", "trees", n_mol=4096, lo=20, hi=200, precision="fp64", start="zero"),
        # a smaller box in float-float precision, with the X-O-H distances of its hydroxyls
        _solve("trees1001_df", "trees", n_mol=1001, lo=20, hi=200, precision="mixed_df", xoh=True),
        # a box of many small molecules
        _solve("small8192_mixed", "trees", n_mol=8192, lo=20, hi=50),
        # a caller that keeps its arrays in page-locked host memory, as the serving loop does
        _solve("trees1000_host", "trees", n_mol=1000, lo=20, hi=200, host=True),
        # one branched molecule of 1400 atoms: the middle of the serving loop's request sizes
        _solve("molecule1400_mixed", "molecule", lo=1400, hi=1400),
        # one protein-like system with bond and H-X-H angle distances: by overlapping domains
        # (the full-size system), and by exact Newton with its Schur complement in float64
        _solve("protein100k_overlap", "protein", lo=100_000, hi=100_000, overlap=4),
        _solve("protein20k_exact", "protein", lo=20_001, hi=20_001, precision="fp64", start="zero"),
        # the learned start of a batch of chains: features and network, one multiplier each
        {"name": "warm_chains4096", "kind": "warm", "n_mol": 4096, "lo": 64, "hi": 64, "topology": 1},
        # one mini-batch of the network's training: forward and backward
        {"name": "gradient8192", "kind": "gradient", "rows": 8192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "trees", "trees", "trees", "molecule", "protein", "warm", "gradient"])
    topology = rng.randrange(1, 1 << 20)
    prec = rng.choice(["mixed", "mixed", "fp64", "mixed_df"])
    start = "zero" if prec == "fp64" else "diag"
    if kind == "chain":
        n = _log_int(rng, 8, 200)
        return _drawn(kind, lo=n, hi=n, topology=topology, precision=prec, start=start)
    if kind == "trees":
        lo, hi = rng.choice([(20, 200), (20, 200), (20, 50), (50, 100)])
        most = {200: 4096, 50: 8192, 100: 4096}[hi]
        return _drawn(kind, n_mol=_log_int(rng, 64, most), lo=lo, hi=hi, topology=topology, precision=prec, start=start,
                      host=rng.random() < 0.2, xoh=rng.random() < 0.25)
    if kind == "molecule":
        n = _log_int(rng, 300, 4000)
        return _drawn(kind, lo=n, hi=n, topology=topology, precision=prec, start=start)
    if kind == "protein":
        n = _log_int(rng, 6000, 100_000)
        return _drawn(kind, lo=n, hi=n, topology=topology, precision=prec, start=start, overlap=rng.choice([0, 4]),
                      xoh=rng.random() < 0.25)
    if kind == "warm":
        return {"kind": kind, "n_mol": _log_int(rng, 64, 4096), "lo": 64, "hi": 64, "topology": topology}
    return {"kind": kind, "rows": _log_int(rng, 256, 8192)}


def _drawn(kind, **kw):
    c = _solve("", kind, **kw)
    del c["name"]
    return c


# ----------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------
@functools.lru_cache(maxsize=16)
def _system(kind, n_mol, lo, hi, topology, xoh):
    """The case's molecules: who is constrained to whom, target distances, masses, one geometry."""
    if kind in ("chain", "warm"):
        return wl.chain_molecules([lo] * n_mol, seed=topology)
    if kind == "trees":
        return wl.tree_batch(n_mol=n_mol, lo=lo, hi=hi, seed=topology, xoh=xoh)
    if kind == "molecule":
        return wl.tree_molecules_of_sizes([lo], seed=topology)
    return wl.protein_like(n_atoms=lo, seed=topology, xoh=xoh)


def _case_system(case):
    return _system(case["kind"], case["n_mol"], case["lo"], case["hi"], case["topology"], case.get("xoh", False))


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _state(s, seed):
    """(x_old, x_unc, inv_mass, d) of one time step: every molecule turned and moved as a rigid
    body (so the reference positions stay feasible), the unconstrained positions perturbed."""
    dev = _device()
    g = torch.Generator(device=dev).manual_seed(seed)
    x = torch.from_numpy(s.x_old).to(dev)
    ptr = torch.from_numpy(s.mol_atom_ptr).to(dev)
    n_mol = ptr.numel() - 1
    mol = torch.repeat_interleave(torch.arange(n_mol, device=dev), ptr[1:] - ptr[:-1])
    centre = x[ptr[:-1]]  # its first atom
    q = torch.randn(n_mol, 4, dtype=torch.float64, device=dev, generator=g)  # random unit quaternions
    a, b, c, e = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (c * c + e * e), 2 * (b * c - a * e), 2 * (b * e + a * c),
                       2 * (b * c + a * e), 1 - 2 * (b * b + e * e), 2 * (c * e - a * b),
                       2 * (b * e - a * c), 2 * (c * e + a * b), 1 - 2 * (b * b + c * c)], 1).view(n_mol, 3, 3)
    shift = torch.rand(n_mol, 3, dtype=torch.float64, device=dev, generator=g)
    x = (rot[mol] @ (x - centre[mol])[:, :, None])[:, :, 0] + (centre + shift)[mol]
    x_old = x.contiguous()
    noise = torch.randn(x.shape, dtype=torch.float64, device=dev, generator=g)
    x_unc = x_old + s.meta["perturbation_nm"] * noise
    f = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
    return x_old, x_unc, f(s.inv_mass), f(s.d)


def _features64(s, x_old, x_unc, w, d):
    """The 16 features of every constraint (the header of the C ABI defines them) and the scale
    between the network's output and a multiplier, in 64 bits."""
    dev = x_old.device
    i = torch.from_numpy(s.atom_i.astype(np.int64)).to(dev)
    j = torch.from_numpy(s.atom_j.astype(np.int64)).to(dev)
    sv, rv = x_unc[i] - x_unc[j], x_old[i] - x_old[j]
    weight, d2 = w[i] + w[j], d * d
    own = (sv * sv).sum(1) / d2 - 1
    sr = (sv * rv).sum(1)
    f = torch.zeros(len(d), 16, dtype=torch.float64, device=dev)
    f[:, 0], f[:, 1], f[:, 2] = own, sr / d2 - 1, (w[i] - w[j]) / weight
    f[:, 3] = ((sv - rv) ** 2).sum(1) / d2
    # the first two other constraints, by number, at each of the two atoms
    n_c = s.n_constraints
    atom = np.concatenate([s.atom_i, s.atom_j])
    con = np.concatenate([np.arange(n_c), np.arange(n_c)])
    by = np.lexsort((con, atom))
    first = np.searchsorted(atom[by], np.arange(s.n_atoms + 1))
    con, number = con[by], np.arange(n_c)
    for side, ends in enumerate((s.atom_i, s.atom_j)):
        at, end = first[ends], first[ends + 1]
        found = np.zeros(n_c, np.int64)
        slot = np.full((n_c, 2), -1, np.int64)
        for k in range(3):
            here = at + k < end
            other = np.where(here, con[np.minimum(at + k, len(con) - 1)], -1)
            take = here & (other != number) & (found < 2)
            slot[number[take], found[take]] = other[take]
            found += take
        for k in range(2):
            q = 4 + 3 * (2 * side + k)
            has = torch.from_numpy(slot[:, k] >= 0).to(dev)
            o = torch.from_numpy(np.maximum(slot[:, k], 0)).to(dev)
            a = torch.from_numpy(ends.astype(np.int64)).to(dev)
            sign = torch.where((a == i) == (a == i[o]), 1.0, -1.0).double()
            f[:, q] = torch.where(has, own[o], 0.0)
            f[:, q + 1] = torch.where(has, sign * (sv * rv[o]).sum(1) / (d * d[o]), 0.0)
            f[:, q + 2] = torch.where(has, w[a] / weight, 0.0)
    return f, 4 * weight * sr / d2


def _parameters(seed):
    """Network parameters like a trained network's: the constraint's own violation carried
    through both layers (the diagonal guess), and a small random part on every weight."""
    r = np.random.default_rng(seed)
    w1, b1 = 0.05 * r.normal(size=(128, 16)), 0.01 * r.normal(size=128)
    w2, b2 = 0.02 * r.normal(size=(128, 128)), 0.01 * r.normal(size=128)
    w3, b3 = 0.02 * r.normal(size=128), np.zeros(1)
    for u, sign in ((0, 1.0), (1, -1.0)):
        w1[u, 0], w2[u, u], w3[u] = sign, 1.0, sign
    return np.concatenate([v.ravel() for v in (w1, b1, w2, b2, w3, b3)]).astype(np.float32)


def _batch(case, seed):
    """A mini-batch: features of chains in some time step, and multipliers around the diagonal guess."""
    s = _system("chain", -(-case["rows"] // 63), 64, 64, 1, False)
    f, _ = _features64(s, *_state(s, seed))
    f = f[: case["rows"]].float().contiguous()
    g = torch.Generator(device=f.device).manual_seed(seed + 1)
    return f, (f[:, 0] * (1 + 0.1 * torch.randn(len(f), device=f.device, generator=g))).contiguous()


def prepare(case, seed):
    if case["kind"] == "gradient":
        mlp = B.Mlp(max_batch=case["rows"], seed=seed)
        mlp.set_params(_parameters(seed))
        return {"case": case, "mlp": mlp, "batch": _batch(case, seed)}
    s = _case_system(case)
    inputs = _state(s, seed)
    if case["kind"] == "warm":
        topo = B.Topology(s.n_atoms, s.atom_i, s.atom_j)
        mlp = B.Mlp(max_batch=1024, seed=seed)
        mlp.set_params(_parameters(seed))
        return {"case": case, "mlp": mlp, "topo": topo, "inputs": inputs}
    if case["host"]:
        inputs = tuple(t.cpu().pin_memory() for t in inputs)
    return {"case": case, "topo": B.Topology(s.n_atoms, s.atom_i, s.atom_j, overlap=case["overlap"]), "inputs": inputs}


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        return state["mlp"].gradient(*state["batch"])
    if case["kind"] == "warm":
        return B.warm_start(state["mlp"], state["topo"], *state["inputs"])
    start = None if case["start"] == "zero" else case["start"]
    x, lam, iterations, status = state["topo"].solve(*state["inputs"], tol=TOL, precision=case["precision"], start=start)
    return {"x": x, "lambda": lam, "iterations": iterations, "status": status}


def work(case):
    if case["kind"] == "gradient":
        n, p = case["rows"], 18817
        # forward, and twice that for the gradients towards inputs of layer 2 and the weights
        return {"bytes": 4 * (17 * n + 2 * p), "flops": 6 * n * (16 * 128 + 128 * 128 + 128)}
    s = _case_system(case)
    n, c, m = s.n_atoms, s.n_constraints, s.n_molecules
    if case["kind"] == "warm":  # positions, masses, distances and pairs in, multipliers out
        return {"bytes": 56 * n + (8 + 8 + 4) * c, "flops": 2 * c * (16 * 128 + 128 * 128 + 128)}
    # positions twice, masses, distances and pairs in; positions, multipliers, iterations and
    # status out.  Per constraint and Newton step: violation, row of the matrix, elimination and
    # substitution, multiplier and position update (about 150 operations), in three steps or
    # four (from a zero start)
    return {"bytes": 80 * n + 24 * c + 8 * m, "flops": 150 * c * (4 if case["start"] == "zero" else 3)}


# ----------------------------------------------------------------------------------
# what the outputs are in 64 bits
# ----------------------------------------------------------------------------------
def _newton64(s, x_old, x_unc, w, d):
    """The multipliers and positions that satisfy every constraint: Newton's method to rounding,
    its linear systems by preconditioned BiCGSTAB on the unassembled matrix G(x) M^-1 G(x_old)^T."""
    dev = x_old.device
    i = torch.from_numpy(s.atom_i.astype(np.int64)).to(dev)
    j = torch.from_numpy(s.atom_j.astype(np.int64)).to(dev)
    rho = x_old[i] - x_old[j]

    def displacement(v):  # M^-1 G(x_old)^T v
        t = (2 * v)[:, None] * rho
        g = torch.zeros_like(x_old).index_add_(0, i, t).index_add_(0, j, -t)
        return w[:, None] * g

    lam = torch.zeros_like(d)
    for _ in range(12):
        x = x_unc - displacement(lam)
        r = x[i] - x[j]
        sigma = (r * r).sum(1) - d * d
        if float((sigma.abs() / (d * d)).max()) < 1e-14:
            break
        diag = 4 * (w[i] + w[j]) * (r * rho).sum(1)

        def apply(v):
            u = displacement(v)
            return 2 * (r * (u[i] - u[j])).sum(1)

        z = sigma / diag
        res = sigma - apply(z)
        shadow, p, ap = res.clone(), res.clone(), None
        rho_k, first = torch.dot(shadow, res), float(res.norm())
        for _ in range(200):
            if float(res.norm()) <= 1e-12 * max(first, float(sigma.norm())) or first == 0:
                break
            y = p / diag
            ap = apply(y)
            alpha = rho_k / torch.dot(shadow, ap)
            half = res - alpha * ap
            h = half / diag
            t = apply(h)
            omega = torch.dot(t, half) / torch.dot(t, t)
            z = z + alpha * y + omega * h
            res = half - omega * t
            new = torch.dot(shadow, res)
            p = res + (new / rho_k) * (alpha / omega) * (p - omega * ap)
            rho_k = new
        lam = lam + z
    return x_unc - displacement(lam), lam


def _network64(theta, f):
    """(first and second hidden layer, output): the weights of both layers, the features and the
    first hidden layer in bfloat16, as the network is defined; everything else in 64 bits."""
    half = lambda v: v.float().bfloat16().double()  # noqa: E731
    w1, b1, w2, b2, w3, b3 = theta.split([2048, 128, 16384, 128, 128, 1])
    h1 = half(torch.relu(half(f) @ half(w1.view(128, 16)).T + b1))
    h2 = torch.relu(h1 @ half(w2.view(128, 128)).T + b2)
    return h1, h2, h2 @ w3 + b3


def exact(case, seed):
    dev = _device()
    if case["kind"] == "gradient":
        f, t = _batch(case, seed)
        theta = torch.from_numpy(_parameters(seed)).to(dev).double()
        f, t = f.double(), t.double()
        h1, h2, y = _network64(theta, f)
        w2 = theta[2176:2176 + 16384].float().bfloat16().double().view(128, 128)
        dy = 2 * (y - t) / len(t)
        dz2 = dy[:, None] * theta[-129:-1] * (h2 > 0)
        dz1 = (dz2 @ w2) * (h1 > 0)
        grad = [dz1.T @ f, dz1.sum(0), dz2.T @ h1, dz2.sum(0), h2.T @ dy, dy.sum().view(1)]
        return torch.cat([v.reshape(-1) for v in grad]), ((y - t) ** 2).mean().view(1)
    s = _case_system(case)
    inputs = _state(s, seed)
    if case["kind"] == "warm":
        f, scale = _features64(s, *inputs)
        return _network64(torch.from_numpy(_parameters(seed)).to(dev).double(), f)[2] / scale
    x, lam = _newton64(s, *inputs)
    return {"x": x, "lambda": lam, "iterations": None, "status": None}
