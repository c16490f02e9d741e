"""Order of a staged long sum's batches (host side, no GPU).

The team's threads meet at barriers only, so between two of them no thread may
read a slot of the offset tables or a half of the element buffer that another
one may be writing, and every read finds the batch it is for."""

import ctypes

import pytest

from paper_1709_03636_gb300 import _lib


@pytest.mark.parametrize("fold_every", [1, 2, 16, 1 << 20])
@pytest.mark.parametrize("n_batches", [1, 2, 3, 4, 5, 8, 33])
def test_no_thread_overtakes_another(n_batches, fold_every):
    faults = ctypes.c_int32(-1)
    _lib.check(_lib.lib.qtc_selftest_stage_schedule(n_batches, fold_every, ctypes.byref(faults)))
    assert faults.value == 0
