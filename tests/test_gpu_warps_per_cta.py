"""Warps per CTA of a small batch, from the networks and the device's SMs: four, halved
while every CTA still has an SM of its own."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402
from synth import random_regular_graph  # noqa: E402


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("sixths", [1, 6, 7, 12, 13, 24])   # of the SMs, in networks
def test_warps_per_cta(sixths, dtype):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = max(6, 2 * (sms * sixths // 18))                    # 3-regular: 1.5 n networks
    batch = q.Batch(q.Circuit.qaoa(n, random_regular_graph(n, 3, n), 1))
    networks, teams = len(batch.edges), 4
    while teams > 1 and 2 * networks <= sms * teams:
        teams //= 2
    info = batch.launch_info(q.Engine(0, arena_bytes=64 << 20), dtype, True)
    assert info["block"] == 32 * teams
    assert info["grid"] == -(-networks // teams)
