"""Length of the single-precision chains behind a complex64 state vector's <C>.

With gamma = 0 every amplitude goes through the same operations, so all probabilities are
one number p, and the edge (0, 1) adds it or nothing: a chain of k additions of p rounds
the same way in every thread, by 1e-5 for 800 terms at these angles and by less than 1e-6
for 432, the most that a thread adds up for n = 26 (16 amplitudes of each of 27 tiles).
Both are emulated here; a further 2^-21 covers p's own rounding (two products and their
sum, contracted or not)."""

from fractions import Fraction
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402

F = np.float32


def fma(a, b, c):
    return F(float(Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c))))


def chain_error(p, terms):
    total = F(0)
    for _ in range(terms):
        total = F(total + p)
    return abs(float(total) / (terms * float(p)) - 1)


@pytest.mark.parametrize("beta", [0.61, 0.421])
def test_expectation_adds_short_chains(beta):
    n = 26
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-(1 << (n - 13)) // (2 * sms))          # of the busiest thread
    r, x, y = F(math.tan(beta)), F(2.0 ** (-n / 2)), F(0)
    for _ in range(n):
        x, y = fma(r, y, x), fma(-r, x, y)
    p = fma(x, x, F(y * y))
    bound = max(chain_error(p, 16 * t) for t in (tiles - 1, tiles)) + 2.0 ** -21
    assert chain_error(p, 32 * tiles) > 4 * bound     # twice the length would show
    exact = math.cos(beta) ** (2 * n) * float(p) * 2.0 ** (n - 1)
    engine = q.Engine(0, arena_bytes=(8 << n) + (64 << 20))
    C, _ = q.statevector_expectation(engine, q.Circuit.qaoa(n, [(0, 1)], 1), [0.0], [beta], "c64")
    assert abs(C / exact - 1) < bound
