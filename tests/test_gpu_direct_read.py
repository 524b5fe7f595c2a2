"""Which host buffers a read's kernel stores into (needs the driver; launches nothing):
only a range that one page-locked allocation or registration holds from end to end."""
import mmap

import pytest

from paper_1810_09299_gb300 import lbm

pytestmark = pytest.mark.gpu
PAGE = 1 << 16  # a multiple of the host's page size (4 KB or 64 KB)


def test_only_ranges_inside_one_registration():
    torch = pytest.importorskip("torch")
    direct = lbm.lib().lbm_selftest_direct_read
    pinned = torch.zeros(1024, dtype=torch.float64, pin_memory=True)
    assert direct(pinned.data_ptr(), 8192) == 1
    assert direct(pinned.data_ptr() + 4, 8) == 0  # not aligned
    assert direct(pinned.data_ptr(), 0) == 0
    pages = torch.frombuffer(mmap.mmap(-1, 8 * PAGE), dtype=torch.uint8)
    at = pages.data_ptr() + -pages.data_ptr() % PAGE
    rt = torch.cuda.cudart()
    assert direct(at, 8) == 0  # pageable
    held = [at, at + 2 * PAGE, at + 3 * PAGE]
    for p in held:
        assert int(rt.cudaHostRegister(p, PAGE, 0)) == 0
    try:
        assert direct(at, PAGE) == 1 and direct(at + PAGE - 8, 8) == 1
        assert direct(at, PAGE + 8) == 0                # past the end
        assert direct(at + 8, 3 * PAGE - 16) == 0       # both ends page-locked, the page between them not
        assert direct(at + 2 * PAGE, 2 * PAGE) == 0     # two registrations side by side
        assert direct(at + PAGE, 8) == 0                # the gap
    finally:
        for p in held:
            rt.cudaHostUnregister(p)
