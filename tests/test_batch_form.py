"""Which batches are built by device-wide sorts (host logic, no GPU): none that the sort would refuse."""
import ctypes

import numpy as np
import pytest

from paper_2601_05347_gb300 import _build, psi

INVALID = 1
P = ctypes.c_void_p(1 << 20)  # never dereferenced: the size is refused first


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


def test_no_batch_that_the_sort_refuses():
    limit = (1 << 30) - 1
    assert psi.lib().psi_test_sort_withheld_tile(P, P, limit, 0, 1, None) == INVALID
    for total in (limit, limit + 1, (1 << 32) - 1):
        assert not psi.batch_device_wide([0, total])
    assert psi.batch_device_wide([0, limit - 1])


@pytest.mark.parametrize("kw,wide", [({}, True), ({"dim": 3, "kind": "spac_z"}, True), ({"coord_bits": 31}, True),
                                     ({"threads": 512}, False), ({"radix_bits": 8}, False),
                                     ({"radix_bits": 11, "threads": 256}, False)])
def test_only_where_the_form_is_left_open(kw, wide):
    assert psi.batch_device_wide(np.array([0, 7, 1_000_007]), **kw) == wide
    assert not psi.batch_device_wide([0, 7, 1007], **kw)
    assert not psi.batch_device_wide([0, 0], **kw)
