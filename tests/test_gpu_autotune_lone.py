"""The autotuner on a molecule that is partitioned below the threshold of overlapping domains: no
overlap depth is tried, since each would be the same plan under another name."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_13075_gb300 import binding as B  # noqa: E402
from paper_2503_13075_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,candidates", [({}, 1), ({"partition_min_constraints": 1200}, 5)])
def test_overlap_depths_only_past_the_domain_threshold(kw, candidates):
    s = wl.chain_molecules([1400], seed=3)
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, **kw)
    assert t.export_layout(0)["n_parts"] > 1
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    tun = t.autotune(f(s.x_old), f(s.x_unc), f(s.inv_mass), f(s.d), reps=2)
    assert tun["candidates"] == candidates
    if candidates == 1:
        assert tun["chosen"]["overlap"] == 0
