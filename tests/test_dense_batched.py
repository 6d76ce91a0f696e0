"""Batched molecules with many terms: a centre bonded to k atoms has a full factor (k^3 / 6 terms).
The program's words hold 16384 pairs of terms: stars of up to 57 bonds stay on the batched kernel,
larger ones take a CTA of their own.
"""
import numpy as np
import pytest

from paper_2503_13075_gb300 import binding as B
from paper_2503_13075_gb300 import workloads as wl


def stars(sizes, seed=2):
    rng = np.random.default_rng(seed)
    mols = []
    for k in sizes:
        z = 1.0 - 2.0 * (np.arange(k) + 0.5) / k
        phi = np.arange(k) * 2.399963
        u = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], 1)
        mols.append((["S"] + ["C"] * k, [(0, a, 0.14) for a in range(1, k + 1)], np.concatenate([np.zeros((1, 3)), 0.14 * u])))
    return wl._exact_lengths(wl._assemble("stars", mols, rng, 0.002, seed, 5.0))


def test_route_of_dense_molecules():
    for k, batched in ((40, True), (47, True), (52, True), (57, True), (58, False), (60, False)):
        s = stars([k])
        t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, plan_only=True)
        assert t.n_large == (0 if batched else 1), k


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_df"])
def test_dense_molecules_solve(prec):
    torch = pytest.importorskip("torch")
    from oracle import ilves_oracle as orc

    s = stars([44, 46, 48, 52, 60])
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j)
    assert t.n_large == 1
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ref = orc.solve_system(s, tol=1e-12)
    x, lam, it, st = (v.cpu().numpy() for v in t.solve(f(s.x_old), f(s.x_unc), f(s.inv_mass), f(s.d), precision=prec))
    assert np.all(st == B.CONVERGED) and np.abs(it - ref.iterations).max() <= 1
    assert np.abs(x - ref.x).max() <= 1e-10
    assert np.all(np.abs(lam - ref.lam) <= 1e-8 * np.abs(ref.lam) + 1e-10 * np.abs(ref.lam).max())
    assert orc.max_relative_violation(x, s.atom_i, s.atom_j, s.d) <= 1e-12
