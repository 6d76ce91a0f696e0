"""The automatic route of a topology's only molecule past the batched kernel's limits, between
1000 and 4095 constraints: partitioned over CTAs where that is the faster side, one CTA where it
is not (few constraints per separator level, grids with dense separators), and where several
such molecules share a launch.  Host plans; the GPU test solves one molecule of each route.
"""
import time

import numpy as np
import pytest

from paper_2503_13075_gb300 import binding as B
from paper_2503_13075_gb300 import workloads as wl


def grid(nx, ny, nz, seed=1):
    """Atoms on a grid, every neighbour distance constrained."""
    idx = np.arange(nx * ny * nz).reshape(nx, ny, nz)
    bonds = [(a, b, 0.15) for p, q in ((idx[:-1], idx[1:]), (idx[:, :-1], idx[:, 1:]), (idx[:, :, :-1], idx[:, :, 1:]))
             for a, b in zip(p.ravel().tolist(), q.ravel().tolist())]
    rng = np.random.default_rng(seed)
    pos = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1).reshape(-1, 3) * 0.15
    pos = pos + rng.normal(0, 0.01, pos.shape)
    return wl._exact_lengths(wl._assemble("grid", [(["C"] * len(pos), bonds, pos)], rng, 0.001, seed, 5.0))


def parts(s, **kw):
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, plan_only=True, **kw)
    big = int(np.argmax(t.molecules()[1]))
    return t.export_layout(big)["n_parts"]


def test_threshold_and_number_of_molecules():
    assert parts(wl.chain_molecules([1000], seed=3)) == 0  # 999 constraints
    assert parts(wl.chain_molecules([1001], seed=3)) > 1  # 1000
    assert parts(wl.chain_molecules([1400, 1400], seed=3)) == 0
    assert parts(wl.chain_molecules([1400] + [50] * 20, seed=3)) > 1  # beside batched molecules
    assert parts(wl.chain_molecules([1400, 300], seed=3)) == 0  # 299 constraints: also on a CTA
    s = wl.chain_molecules([2000], seed=3)
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, plan_only=True, overlap=2)
    assert t.export_domains(0)["cons"] == [] and t.export_layout(0)["n_parts"] > 1  # no domains below 4096
    assert parts(s, partition_min_constraints=3000) == 0


def test_separator_levels_decide():
    # trees of 1002 atoms whose parts leave 7 and 11 levels of separators
    assert parts(wl.tree_molecules_of_sizes([1002], seed=1)) > 1
    assert parts(wl.tree_molecules_of_sizes([1002], seed=2)) == 0
    for n in (1400, 2000, 4000):
        assert parts(wl.tree_molecules_of_sizes([n], seed=3)) > 1
    assert parts(wl.protein_like(2000, seed=3, xoh=True)) > 1


def test_dense_separators_stay_on_one_cta():
    assert parts(grid(24, 24, 1)) == 0
    assert parts(grid(150, 8, 1)) > 1  # 40 levels of separators, but a tenth of the terms
    s = grid(2, 2, 300)  # cut across: 849 levels, whose plan alone took half a minute
    t0 = time.perf_counter()
    assert parts(s) == 0
    auto = time.perf_counter() - t0
    t0 = time.perf_counter()
    parts(s, partition_min_constraints=1 << 30)
    assert auto < 5 * (time.perf_counter() - t0) + 1.0


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_df"])
@pytest.mark.parametrize("case", ["tree", "grid"])
def test_lone_molecule_solves(case, prec):
    torch = pytest.importorskip("torch")
    from oracle import ilves_oracle as orc

    s = wl.tree_molecules_of_sizes([1400], seed=1) if case == "tree" else grid(8, 8, 8)
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j)
    assert (t.export_layout(0)["n_parts"] > 1) == (case == "tree")
    # no more than the one-CTA path took of the static scratch
    one = B.Topology(s.n_atoms, s.atom_i, s.atom_j, partition_min_constraints=1 << 30)
    assert t.workspace_bytes() <= max(2 * one.workspace_bytes(), 1 << 20)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    args = (f(s.x_old), f(s.x_unc), f(s.inv_mass), f(s.d))
    ref = orc.solve_system(s, tol=1e-12)
    for solve in (t.solve, t.solve_static_scratch):
        x, lam, it, st = (v.cpu().numpy() for v in solve(*args, precision=prec))
        assert np.all(st == B.CONVERGED) and np.abs(it - ref.iterations).max() <= 1
        assert np.abs(x - ref.x).max() <= 1e-10
        assert np.all(np.abs(lam - ref.lam) <= 1e-8 * np.abs(ref.lam) + 1e-10 * np.abs(ref.lam).max())
        assert orc.max_relative_violation(x, s.atom_i, s.atom_j, s.d) <= 1e-12
