"""Which steps of the graph executor are staged long sums, and their emulation on the
host (no GPU): the networks of test_gpu_staged_sums reach every order of addition, in
forward and adjoint steps and beyond 4096 values."""

import ctypes

import pytest

import paper_1709_03636_gb300 as q
from paper_1709_03636_gb300 import _lib
from synth import random_regular_graph

# n, degree, p, diagonal gates, ordering, largest rank in shared memory
CASES = [(14, 5, 1, False, "stoch", 3), (13, 4, 2, False, "stoch", 4)]


def batch_of(n, d, p, diag, ordering, small_rank):
    edges = random_regular_graph(n, d, n + d)
    return q.Batch(q.Circuit.qaoa(n, edges, p), lightcone=False, diag=diag, ordering=ordering,
                   seed=1)


def staged(batch, dtype, grad, small_rank):
    """Staged steps: sequential, eight accumulators, four of pairs; beyond 4096 values."""
    counts = (ctypes.c_int32 * 4)()
    _lib.check(_lib.lib.qtc_selftest_stage_steps(batch.ptr, q.DTYPES[dtype], int(grad), 1,
                                                 small_rank, counts))
    return list(counts)


def test_every_order_is_reached():
    # complex64 / complex128 (which has no pairs): together, value and gradient of the
    # whole batches and of their middle networks alone
    for dtype, orders in (("c64", (0, 1, 2, 3)), ("c128", (0, 1))):
        forward, adjoint = [0] * 4, [0] * 4
        for case in CASES:
            batch = batch_of(*case)
            for b in (batch, batch.subset([len(batch.edges) // 2])):
                f, g = staged(b, dtype, False, case[-1]), staged(b, dtype, True, case[-1])
                forward = [x + y for x, y in zip(forward, f)]
                adjoint = [x + y - z for x, y, z in zip(adjoint, g, f)]
        assert all(forward[k] > 0 for k in orders), (dtype, forward)
        assert all(adjoint[k] > 0 for k in orders), (dtype, adjoint)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("case", CASES)
def test_emulated_steps_equal_the_plain_contraction(case, dtype):
    batch = batch_of(*case)
    one = batch.subset([len(batch.edges) // 2])
    trees = one.execution_trees(dtype)
    for b in (one, trees):
        err, count = ctypes.c_double(), ctypes.c_int32()
        _lib.check(_lib.lib.qtc_selftest_tile_steps(b.ptr, q.DTYPES[dtype], 1, 1, case[-1], 0, 18,
                                                    ctypes.byref(err), ctypes.byref(count)))
        assert count.value > 0
        assert err.value < 1e-11
