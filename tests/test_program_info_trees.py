"""program_info describes the program that an engine runs (host side, no GPU).

The graph executor contracts complex128 networks along rearranged trees that move less:
their tensors in global memory take less than twice those of single precision, which
runs the plans' own (the same elements of half the size)."""

import pytest

import paper_1709_03636_gb300 as q
from synth import random_regular_graph


@pytest.mark.parametrize("grad", [False, True])
def test_complex128_programs_run_the_execution_trees(grad):
    n = 18
    batch = q.Batch(q.Circuit.qaoa(n, random_regular_graph(n, 7, 2), 1), lightcone=False)
    single = batch.program_info("c64", grad)
    double = batch.program_info("c128", grad)
    assert single["graph"] and double["graph"]
    assert double["net_global_bytes_unshared"] < 1.8 * single["net_global_bytes_unshared"]
    own = batch.stats()["cmacs"]
    assert batch.execution_trees("c64").stats()["cmacs"] == own
    assert batch.execution_trees("c128").stats()["cmacs"] < 0.9 * own


def test_a_tight_shared_memory_limit_takes_the_plans_own_tree():
    """A rearranged tree may need a larger subtree arena than the plan's own: where a CTA
    has no room for it, the network keeps the plan's, as single precision does anywhere."""
    n = 16
    edges = random_regular_graph(n, 3, n)
    batch = q.Batch(q.Circuit.qaoa(n, edges, 1), edges[:4], lightcone=False, ordering="stoch")
    free = batch.program_info("c128", True, force_graph=True)["smem_bytes"]
    for limit in (free, 44000, 40000):
        info = batch.program_info("c128", True, force_graph=True, smem_limit=limit + 16384)
        assert info["graph"] and info["smem_bytes"] <= limit
    assert free > 44000
