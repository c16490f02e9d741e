"""Sums over the leaves of one parameter in the graph executor are taken in FP64,
in every element type.

The amplitude <0..0| RZ(c t)^k |0..0> at t = 0 is one, every intermediate holds ones
and zeros, and each of the k leaves contributes exactly -i c / 2 to the derivative in
either precision.  So only the sum over leaves rounds: k 2^-53 relative in FP64
(1.4e-13 for 1200 leaves), against k 2^-24 for a chain in FP32."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("diag", [True, False])
@pytest.mark.parametrize("n,k,n_params", [(3, 400, 1), (2, 150, 4), (1, 700, 6), (4, 300, 8),
                                          (2, 300, 9)])
def test_equal_terms_add_up_in_fp64(n, k, n_params, diag, dtype):
    c = float(np.float32(0.7))
    circ = q.Circuit(n, n_params)
    count = [0] * n_params
    for i in range(k):
        for v in range(n):
            slot = (i * n + v) % n_params
            circ.add_gate("rz", [v], slot=slot, coeff=c)
            count[slot] += 1
    plan = q.Plan(q.Network(circ, "amplitude", bits=[0] * n, lightcone=False, diag=diag), "lg")
    engine = q.Engine(0, arena_bytes=256 << 20)
    engine.set_graph_options(True, 4)
    value, grad = q.contract(engine, plan, [0.0] * n_params, dtype, want_grad=True)
    assert value == 1.0
    for got, m in zip(grad, count):
        assert abs(got - (-0.5j * c * m)) < 1e-12 * c * m
