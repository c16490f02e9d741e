"""<Z_a Z_b> of a state vector against the exact sums over the state that the device holds.

A state of 2^12 amplitudes is one tile, which the per-edge pass leaves as it is at the end
of the arena.  Probabilities and signed sums are FP64 in either element type.  Rounding
errors of the tree of additions, as independent uniform ones on the masses it adds (256
threads of mass 2^-8, eight of them per lane, five levels over the lanes), come to 0.45
2^-53 rms; the bound is 2^-53 rms over all edges and angles and 30 2^-53 for any one."""

import random

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402
from synth import random_regular_graph  # noqa: E402


@pytest.mark.parametrize("dtype,kind", [("c64", np.complex64), ("c128", np.complex128)])
@pytest.mark.parametrize("d,p", [(3, 1), (5, 2), (8, 3)])
def test_per_edge_values_are_fp64_sums_of_the_stored_state(dtype, kind, d, p):
    n = 12
    edges = sorted(tuple(sorted(e)) for e in random_regular_graph(n, d, d + p))
    circ = q.Circuit.qaoa(n, edges, p)
    engine = q.Engine(0, arena_bytes=64 << 20)
    x = np.arange(1 << n)
    sign = [1 - 2 * (((x >> u) ^ (x >> v)) & 1) for u, v in edges]
    rng, errors = random.Random(d), []
    for _ in range(20):
        g = [rng.uniform(0, 3.1) for _ in range(p)]
        b = [rng.uniform(0, 1.5) for _ in range(p)]
        _, zz = q.statevector_expectation(engine, circ, g, b, dtype, per_edge=True)
        psi = engine.arena[-(np.dtype(kind).itemsize << n):].cpu().numpy().view(kind)
        prob = psi.real.astype(np.longdouble) ** 2 + psi.imag.astype(np.longdouble) ** 2
        assert abs(float(prob.sum()) - 1) < 1e-5
        errors += [float(np.longdouble(z) - (prob * s).sum()) for z, s in zip(zz, sign)]
    errors = np.array(errors)
    assert np.max(np.abs(errors)) < 30 * 2.0 ** -53
    assert np.sqrt(np.mean(errors ** 2)) < 2.0 ** -53
