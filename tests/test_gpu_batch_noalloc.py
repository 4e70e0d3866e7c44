"""A batch takes its memory when it is created and when query room is reserved: building it, by a block per index or by
device-wide sorts, takes none from the device's memory pool, so it cannot run out of memory half-way or leave allocation
nodes in a captured graph."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2601_05347_gb300 import gen  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi

USED_NOW, USED_HIGH = 7, 8  # CUmemPool_attribute


class PoolHigh:
    """Bytes by which the default memory pool's use rose, at most, inside the block."""

    def __enter__(self):
        self.cu, self.pool = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
        dev = ctypes.c_int(0)
        assert self.cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), dev) == 0
        torch.cuda.synchronize()
        zero = ctypes.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.pool, USED_HIGH, ctypes.byref(zero)) == 0
        self.before = self.get(USED_NOW)
        return self

    def get(self, attr):
        v = ctypes.c_uint64(0)
        assert self.cu.cuMemPoolGetAttribute(self.pool, attr, ctypes.byref(v)) == 0
        return v.value

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        self.rise = self.get(USED_HIGH) - self.before


def batch(sizes, threads):
    off = np.concatenate([[0], np.cumsum(sizes)])
    pts = torch.from_numpy(gen.uniform(int(off[-1]), 2, 30, 7)).to("cuda")
    return psi.Batch(off, dim=2, kind="spac_h", threads=threads), pts, torch.arange(len(pts), dtype=torch.int32,
                                                                                    device="cuda")


@pytest.mark.parametrize("threads", [0, 512])
@pytest.mark.parametrize("sizes", [[30000], [90000, 5], [80000, 0, 700]])  # both tile sizes of the sorts
def test_build_takes_no_memory(sizes, threads):
    b, pts, ids = batch(sizes, threads)
    with PoolHigh() as m:
        n0 = psi.launch_count()
        b.build(pts, ids)
    assert (psi.launch_count() - n0 > 1) == (threads == 0)  # the form that was meant
    assert m.rise == 0
    b.sync()


@pytest.mark.parametrize("reserved,asked", [(80001, 80000), (80001, 500), (200_000, 200_000), (200_000, 33)])
def test_knn_takes_no_memory(reserved, asked):
    b, pts, ids = batch([30000, 9], 0)
    b.build(pts, ids)
    b.reserve(reserved)
    q = pts[torch.arange(asked, device="cuda") % len(pts)].contiguous()
    qoff = torch.tensor([0, asked, asked], device="cuda")
    for k in (10, 40):
        out = torch.empty((asked, k), dtype=torch.int32, device="cuda"), torch.empty((asked, k), dtype=torch.int64,
                                                                                      device="cuda")
        with PoolHigh() as m:
            b.knn(q, qoff, k, *out)
        assert m.rise == 0
    b.sync()
