"""Staged long sums of the graph executor.

A network's steps are staged or cut differently when it runs alone and in a batch; a
forward sum is added in the same order either way, so the values are equal bit for bit.
Against the state vector: the bounds of the element types (complex128 1e-11, complex64
2e-6 per edge and 1e-4 relative on the gradient, here summed over networks that run alone,
whose adjoint sums are staged too)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402
from oracle import statevector as sv  # noqa: E402
from synth import random_regular_graph  # noqa: E402
from test_staged_sums import CASES, batch_of, staged  # noqa: E402


@pytest.mark.parametrize("dtype,tol,gtol", [("c128", 1e-11, 1e-9), ("c64", 2e-6, 1e-4)])
@pytest.mark.parametrize("case", CASES)
def test_alone_and_in_a_batch(case, dtype, tol, gtol):
    n, d, p, _, _, small_rank = case
    batch = batch_of(*case)
    m = len(batch.edges)
    g, b = [0.45 + 0.3 * k for k in range(p)], [0.85 - 0.2 * k for k in range(p)]
    edges = random_regular_graph(n, d, n + d)
    ref = sv.edge_zz(n, edges, g, b)
    _, ref_grad = sv.gradient(n, edges, g, b)
    engine = q.Engine(0, arena_bytes=12 << 30)
    engine.set_graph_options(True, small_rank)
    assert sum(staged(batch, dtype, False, small_rank)[:3]) > 0
    _, zz, _ = q.qaoa_expectation(engine, batch, g, b, dtype)
    assert np.max(np.abs(np.array(zz) - ref)) < tol
    total = np.zeros(2 * p)
    for i in range(m):
        one = batch.subset([i])
        _, alone, _ = q.qaoa_expectation(engine, one, g, b, dtype)
        assert alone[0] == zz[i]
        _, again, grad = q.qaoa_expectation(engine, one, g, b, dtype, want_grad=True)
        assert again[0] == zz[i]
        total += grad
    assert np.max(np.abs(total - ref_grad)) < gtol * max(1, np.max(np.abs(ref_grad)))
