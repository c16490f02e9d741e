"""A program prepared in one engine's arena is never taken for another engine's, also when
the next engine comes to lie at the address of one that has ended."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402
from synth import random_regular_graph  # noqa: E402


def test_the_next_engine_prepares_its_own_program():
    batch = q.Batch(q.Circuit.qaoa(20, random_regular_graph(20, 3, 0), 1))
    for _ in range(8):
        engine = q.Engine(0, arena_bytes=16 << 20)
        batch.prepare(engine, "c64")
        engine.close()
        small = q.Engine(0, arena_bytes=4096)
        with pytest.raises(q.QtcError, match="ARENA"):
            batch.prepare(small, "c64")
        small.close()


def test_the_next_engine_sets_up_its_own_state_vector():
    circ = q.Circuit.qaoa(10, random_regular_graph(10, 3, 0), 1)
    for _ in range(8):
        engine = q.Engine(0, arena_bytes=16 << 20)
        C, _ = q.statevector_expectation(engine, circ, [0.4], [0.3], "c128")
        assert 0 < C < 15
        engine.close()
        small = q.Engine(0, arena_bytes=1024)
        with pytest.raises(q.QtcError, match="ARENA"):
            q.statevector_expectation(small, circ, [0.4], [0.3], "c128")
        small.close()
