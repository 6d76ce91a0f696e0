"""Molecules that the plan gives to the batched kernel but whose slice does not fit the CTAs'
arenas (four CTAs per SM: 56 KB each) are solved by a CTA of their own, beside smaller ones that
stay batched: same results as the oracle's, with the bounds of every result (test_gpu_parity).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ilves_oracle as orc  # noqa: E402
from paper_2503_13075_gb300 import binding as B  # noqa: E402
from paper_2503_13075_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system():
    s = wl.tree_molecules_of_sizes([30, 256, 244, 100, 252, 250, 60], seed=21)
    return s, orc.solve_system(s, tol=1e-12)


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_df"])
def test_slices_past_the_arena(prec, system):
    s, ref = system
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, ctas_per_sm=4)
    atoms, _, _, first = t.molecules()
    assert t.n_large >= 2 and t.n_large < t.n_molecules  # both kernels run
    for m in range(t.n_molecules):
        gid = t.export_layout(m)["atom_gid"]
        assert sorted(gid) == list(range(first[m], first[m] + atoms[m]))
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    x, lam, it, st = (v.cpu().numpy() for v in t.solve(f(s.x_old), f(s.x_unc), f(s.inv_mass), f(s.d), precision=prec))
    assert np.all(st == B.CONVERGED)
    assert np.abs(it - ref.iterations).max() <= 1
    assert np.abs(x - ref.x).max() <= 1e-10
    assert np.all(np.abs(lam - ref.lam) <= 1e-8 * np.abs(ref.lam) + 1e-10 * np.abs(ref.lam).max())
    assert orc.max_relative_violation(x, s.atom_i, s.atom_j, s.d) <= 1e-12
