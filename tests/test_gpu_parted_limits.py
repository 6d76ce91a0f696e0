"""Partitioned solves with one, two and three CTAs to an SM: the shared memory a CTA may take
depends on it (parts' programs and values in shared memory, or read from global memory)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ilves_oracle as orc  # noqa: E402
from paper_2503_13075_gb300 import binding as B  # noqa: E402
from paper_2503_13075_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system():
    s = wl.protein_like(n_atoms=12000, seed=7)
    return s, orc.solve_system(s, tol=1e-12)


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_df"])
@pytest.mark.parametrize("part,per_sm", [(400, 1), (93, 1), (88, 2), (60, 2), (44, 3), (32, 3)])
def test_ctas_per_sm(part, per_sm, prec, system):
    s, ref = system
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, part_constraints=part)
    n = t.export_layout(0)["n_parts"] + 1  # the separators have a CTA of their own
    if n_sm == 152:
        assert (n + n_sm - 1) // n_sm == per_sm
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    x, lam, it, st = (v.cpu().numpy() for v in t.solve(f(s.x_old), f(s.x_unc), f(s.inv_mass), f(s.d), precision=prec))
    assert st.tolist() == [B.CONVERGED] and np.abs(it - ref.iterations).max() <= 1
    assert np.abs(x - ref.x).max() <= 1e-10
    assert np.all(np.abs(lam - ref.lam) <= 1e-8 * np.abs(ref.lam) + 1e-10 * np.abs(ref.lam).max())
    assert orc.max_relative_violation(x, s.atom_i, s.atom_j, s.d) <= 1e-12
