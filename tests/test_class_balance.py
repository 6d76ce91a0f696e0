"""Slots of the two team classes on batches of mixed sizes with an explicit threshold: the large
molecules keep enough 96-thread slots (1.6 units of time a one-warp team takes per unit of cost;
with 2.2 the last 20 % of the molecules got one slot per CTA)."""
import pytest

from paper_2503_13075_gb300 import binding as B
from paper_2503_13075_gb300 import workloads as wl


@pytest.mark.parametrize("narrow,wide_slots", [(130, 3), (160, 2)])
def test_wide_slots_per_cta(narrow, wide_slots):
    s = wl.tree_batch(4096, 20, 200, seed=1)
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, plan_only=True, narrow_atoms=narrow)
    sc = t.schedule("mixed")
    assert sc["n_slots_wide"] >= wide_slots * 152
    assert (sc["slot_team"] == 32).sum() >= 5 * 152
