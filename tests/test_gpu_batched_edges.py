"""The batched kernel at the edges of its program: molecules of one constraint (no elimination
level), atoms of four to seven constraints (incidences past the fourth), levels of 16, 17, 32
and 33 items or pivots and the widest ones (teams hand the narrow levels to one warp), odd and
even numbers of terms -- on both team widths, in every precision, Newton and ILVES-F.

Bounds as for every result (test_gpu_parity): violation 1e-12, positions 1e-10 nm, multipliers
1e-8 relative, iterations +-1 of the oracle's.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ilves_oracle as orc  # noqa: E402
from paper_2503_13075_gb300 import binding as B  # noqa: E402
from paper_2503_13075_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


def _star(rng, k):
    """A centre bonded to k atoms in directions spread over the sphere."""
    z = 1.0 - 2.0 * (np.arange(k) + 0.5) / k
    phi = np.arange(k) * 2.399963
    u = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], 1)
    q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    pos = np.concatenate([np.zeros((1, 3)), 0.14 * u @ q.T])
    return ["S"] + ["C"] * k, [(0, a, 0.14) for a in range(1, k + 1)], pos


@pytest.fixture(scope="module")
def edges():
    rng = np.random.default_rng(77)
    mols = [wl._chain(rng, n) for n in (2, 3, 4, 17, 18, 33, 34, 35, 64, 65, 66, 97, 129, 200, 256)]
    mols += [_star(rng, k) for k in (2, 4, 5, 6, 7)]
    mols += [wl._with_xoh(wl._tree_molecule(rng, n)) for n in (20, 47, 64, 96, 97, 150, 200)]
    s = wl._exact_lengths(wl._assemble("edges", mols, rng, 0.002, 77, 5.0))
    return s, orc.solve_system(s, tol=1e-12), orc.solve_system(s, tol=1e-12, max_iter=80, method="chord")


@pytest.mark.parametrize("method", ["newton", "chord"])
@pytest.mark.parametrize("narrow", [-1, 255])
@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_df"])
def test_batched_edges(prec, narrow, method, edges):
    s, ref, ref_chord = edges
    t = B.Topology(s.n_atoms, s.atom_i, s.atom_j, narrow_atoms=narrow)
    team = t.schedule(prec)["mol_team"]
    assert t.n_large == 0 and np.all(team[: len(team)] == (96 if narrow < 0 else np.where(t.molecules()[0] <= 255, 32, 96)))
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    for start in (None, "diag"):
        x, lam, it, st = (v.cpu().numpy() for v in t.solve(
            f(s.x_old), f(s.x_unc), f(s.inv_mass), f(s.d), precision=prec, method=method, max_iter=80, start=start))
        assert np.all(st == B.CONVERGED)
        want = (ref if method == "newton" else ref_chord).iterations
        assert np.abs(it - want).max() <= (1 if start is None else 2)
        assert np.abs(x - ref.x).max() <= 1e-10
        assert np.all(np.abs(lam - ref.lam) <= 1e-8 * np.abs(ref.lam) + 1e-10 * np.abs(ref.lam).max())
        # ILVES-F in float-float stops just under the tolerance in its own arithmetic
        slack = 2.0**-44 if (prec, method) == ("mixed_df", "chord") else 0.0
        assert orc.max_relative_violation(x, s.atom_i, s.atom_j, s.d) <= 1e-12 + slack
