"""links_get into a buffer that no one page-locked region holds: refused by the copy, as it always was, and not left to
a kernel's stores, for which pages between two regions may not be there."""
import mmap

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_links_get_across_two_registrations(precision):
    # (the pages between the two registrations are there, so that no kernel could fault on them)
    import torch

    import paper_0904_1179_gb300 as su3
    L = (8, 8, 8, 4)  # 18 x 64 KiB of links
    shape = su3.links_shape(L)
    n = int(np.prod(shape))
    whole = np.frombuffer(mmap.mmap(-1, 8 * n + (1 << 16)), dtype=np.float64)
    whole[:] = -7.0
    out = whole[:n].reshape(shape)
    first, last = out.ctypes.data, out.ctypes.data + 8 * n - (1 << 17)
    cudart = torch.cuda.cudart()
    torch.zeros(1, device="cuda")
    assert int(cudart.cudaHostRegister(first, 1 << 18, 0)) == 0
    assert int(cudart.cudaHostRegister(last, 1 << 17, 0)) == 0
    try:
        with su3.Lattice(L, 5.7, 7, start=su3.SU3_HOT, precision=precision) as lat:
            want = lat.get_links()
            with pytest.raises(su3.Su3Error):
                lat.get_links(out)
            assert (whole == -7.0).all()
            assert np.array_equal(lat.get_links(), want)
    finally:
        cudart.cudaHostUnregister(first)
        cudart.cudaHostUnregister(last)
