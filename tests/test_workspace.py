"""CPU: a plan's workspace stays near what its samples and pixels need, for many short chunks too."""
import ctypes

import numpy as np
import pytest

from paper_1705_01893_gb300 import binding, build


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load()


@pytest.mark.parametrize("n,chunks", [(256, 4000), (1024, 4000), (3000, 1000), (4096, 100), (1 << 15, 100)])
@pytest.mark.parametrize("ncomp", [1, 3])
def test_no_large_share_per_chunk(lib, n, chunks, ncomp):
    """Twice the chunks on the same map take twice the bytes that depend on them.  Per sample: spectrum,
    Nbar and intermediate 10, pointing copy 4 or 12, general tables; per chunk a few records: below
    48 bytes a sample for chunks of 256 samples and more, with the records."""
    size = []
    for c in (chunks, 2 * chunks):
        off = (np.arange(c + 1, dtype=np.int64) * n)
        v = ctypes.c_size_t()
        assert lib.mm_plan_workspace_size(c, off.ctypes.data_as(ctypes.POINTER(ctypes.c_int64)), 1000, ncomp, 0,
                                          ctypes.byref(v)) == binding.MM_OK
        size.append(v.value)
    assert (size[1] - size[0]) / (chunks * n) <= 48
