"""Kernels of the warm-start network that start while the kernel before them still runs.

What the kernel before them writes is not constant for their life, so they may not read it as
such: no ``const __restrict__`` pointer and no ``__ldg`` on it (read-only loads, which the compiler
may also move across the wait).  Shown on the source: on the GPU a wrong order need not show.
The GPU tests run the calls back to back and captured, on inputs that differ from call to call.
"""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_13075_gb300", "csrc")
# inputs of the calls and weights: complete before the first kernel of a chain starts
COMPLETE = {"X", "t", "w2b", "params", "w1", "w2", "F", "xr"}


def _balanced(text, start, pair):
    depth = 0
    for k in range(start, len(text)):
        depth += (text[k] == pair[0]) - (text[k] == pair[1])
        if depth == 0:
            return text[start + 1 : k], k + 1
    raise AssertionError("unbalanced")


def test_dependent_kernels_read_results_as_plain_memory():
    text = open(os.path.join(CSRC, "mlp.cu")).read()
    kernels = {m for m in re.findall(r"launch_after\((k_\w+)", text)}
    assert kernels >= {"k_mlp_forward", "k_mlp_backward", "k_grad_reduce"}
    for name in kernels:
        at = re.search(r"__launch_bounds__\([^)]*\)\s+" + name + r"\(", text).end() - 1
        params, after = _balanced(text, at, "()")
        body, _ = _balanced(text, text.index("{", after), "{}")
        if "wait_for_previous" not in body:
            continue
        for p in params.split(","):
            if "const" in p and "__restrict__" in p:
                assert p.split()[-1] in COMPLETE, (name, p)
        for m in re.finditer(r"__ldg\(", body):
            arg, _ = _balanced(body, m.end() - 1, "()")
            arg = re.sub(r"reinterpret_cast<[^>]*>", "", arg)
            assert re.search(r"[A-Za-z_]\w*", arg).group() in COMPLETE, (name, arg)


@pytest.fixture(scope="module")
def torch_():
    return pytest.importorskip("torch")


def _batches(torch, n, rows, seed):
    rng = np.random.default_rng(seed)
    return [(torch.from_numpy(rng.normal(0, 0.3, (rows, 16)).astype(np.float32)).cuda(),
             torch.from_numpy(rng.normal(size=rows).astype(np.float32)).cuda()) for _ in range(n)]


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [7, 3000, 152 * 200 + 7])
def test_gradients_back_to_back(torch_, rows):
    """Calls in a row on one stream, each on other rows, equal the same calls one at a time."""
    from paper_2503_13075_gb300 import binding as B

    mlp = B.Mlp(max_batch=rows, seed=3)
    batches = _batches(torch_, 4, rows, rows)
    want = []
    for b in batches:
        want.append([v.clone() for v in mlp.gradient(*b)])
        torch_.cuda.synchronize()
    for _ in range(5):
        got = [mlp.gradient(*b) for b in batches]
        torch_.cuda.synchronize()
        for g, w in zip(got, want):
            assert torch_.equal(g[0], w[0]) and torch_.equal(g[1], w[1])
    assert mlp.check() == 0


@pytest.mark.gpu
def test_gradient_and_warm_start_captured(torch_):
    """A captured gradient and a captured learned start, replayed on other inputs, equal eager calls."""
    from paper_2503_13075_gb300 import binding as B
    from paper_2503_13075_gb300 import workloads as wl

    rows = 2049
    mlp = B.Mlp(max_batch=rows, seed=3)
    batches = _batches(torch_, 3, rows, 11)
    s = wl.chain_molecules([64] * 50, seed=4)
    topo = B.Topology(s.n_atoms, s.atom_i, s.atom_j)
    dev = lambda v: torch_.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    x_old, w, d = dev(s.x_old), dev(s.inv_mass), dev(s.d)
    rng = np.random.default_rng(5)
    moved = [dev(s.x_old + rng.normal(0, 0.002, s.x_old.shape)) for _ in range(3)]
    f, t, x_unc = batches[0][0].clone(), batches[0][1].clone(), moved[0].clone()
    mlp.gradient(f, t)
    B.warm_start(mlp, topo, x_old, x_unc, w, d)
    torch_.cuda.synchronize()
    graph = torch_.cuda.CUDAGraph()
    with torch_.cuda.graph(graph):
        g, loss = mlp.gradient(f, t)
        l0 = B.warm_start(mlp, topo, x_old, x_unc, w, d)
    for (fk, tk), xk in zip(batches, moved):
        f.copy_(fk)
        t.copy_(tk)
        x_unc.copy_(xk)
        graph.replay()
        ge, le = mlp.gradient(fk, tk)
        l0e = B.warm_start(mlp, topo, x_old, xk, w, d)
        torch_.cuda.synchronize()
        assert torch_.equal(g, ge) and torch_.equal(loss, le) and torch_.equal(l0, l0e)
    assert mlp.check() == 0
