"""Warp teams per CTA of batches around the number of SMs."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402
from oracle import closed_form as cf  # noqa: E402
from synth import random_regular_graph  # noqa: E402


@pytest.fixture(scope="module")
def engine():
    return q.Engine(0, arena_bytes=256 << 20)


# per_cta: warps per CTA the batch asks for, as networks / SMs rounded up to 1, 2 or 4
@pytest.mark.parametrize("over,per_cta", [(-2, 1), (0, 1), (3, 2), (149, 2), (155, 4), (900, 4)])
@pytest.mark.parametrize("dtype,tol", [("c128", 1e-11), ("c64", 2e-6)])
def test_every_network_runs_whatever_the_warps_per_cta(engine, over, per_cta, dtype, tol):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * ((sms + over) // 3 + (1 if over > 0 else 0))   # 3-regular: 1.5 n networks
    edges = [tuple(sorted(e)) for e in random_regular_graph(n, 3, n)]
    g, b = [0.47], [0.29]
    batch = q.Batch(q.Circuit.qaoa(n, edges, 1))
    C, zz, grad = q.qaoa_expectation(engine, batch, g, b, dtype, want_grad=True)
    if sms == 152 and dtype == "c64":
        assert batch.launch_info(engine, dtype, True)["block"] == 32 * per_cta
    ref = np.array([cf.zz_p1(g[0], b[0], *cf.edge_params(n, edges, e)) for e in edges])
    assert np.max(np.abs(np.array(zz) - ref)) < tol
    assert abs(C - cf.maxcut_p1(n, edges, g[0], b[0])) < tol * len(edges)
    want = np.array(cf.maxcut_p1_grad(n, edges, g[0], b[0]))
    assert np.max(np.abs(np.array(grad) - want)) < 10 * tol * len(edges)
