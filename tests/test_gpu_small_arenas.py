"""Arenas that are too small for the faster form of a program take its smallest one.

The tables of the form that runs otherwise are `table_bytes`; the smallest arena that a
batch is accepted in has less than that beside its work buffer, and gives the same
values: bit for bit without a gradient (forward sums keep their order), and to rounding
with it."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402
from synth import random_regular_graph  # noqa: E402


@pytest.mark.parametrize("dtype,tol", [("c64", 2e-5), ("c128", 1e-11)])
@pytest.mark.parametrize("n,d,p,diag,grad,graph", [
    (24, 4, 2, False, False, True),    # subtree tasks and staged sums
    (24, 4, 2, False, True, True),     # the same with leaf dots
    (20, 3, 2, False, True, False),    # one network per CTA
    (20, 3, 2, False, False, False),
])
def test_smallest_arena(n, d, p, diag, grad, graph, dtype, tol):
    edges = random_regular_graph(n, d, n)
    g, b = [0.4 + 0.3 * k for k in range(p)], [0.7 - 0.2 * k for k in range(p)]
    batch = q.Batch(q.Circuit.qaoa(n, edges, p), diag=diag)

    def engine(size):
        e = q.Engine(0, arena_bytes=size)
        e.set_graph_options(graph, 6 if graph else 0)
        return e

    big = engine(1 << 30)
    C, zz, slopes = q.qaoa_expectation(big, batch, g, b, dtype, want_grad=grad)
    low, high = 0, 1 << 20       # refused, accepted, in units of 1 KB
    while high - low > 1:
        mid = (low + high) // 2
        try:
            batch.prepare(engine(mid << 10), dtype, want_grad=grad)
            high = mid
        except q.QtcError as err:
            assert "ARENA" in str(err)
            low = mid
    info = batch.program_info(dtype, grad, force_graph=graph, small_rank=6 if graph else 0)
    assert not info["warp_teams"]
    assert (high << 10) - info["work_bytes"] < 0.95 * info["table_bytes"]
    C2, zz2, slopes2 = q.qaoa_expectation(engine(high << 10), batch, g, b, dtype, want_grad=grad)
    if grad:
        assert abs(C2 - C) <= tol * len(edges)
        assert np.max(np.abs(np.array(slopes2) - slopes)) <= tol * len(edges)
    else:
        assert zz2 == zz
