"""links_get into page-locked memory (the conversion kernel writes it), into page-locked memory off a 16-byte boundary
and into pageable memory (both through the staging buffer): the same bytes, nothing written past the buffer's ends."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _buffer(shape, pinned, skip):
    """A buffer of `shape` that starts `skip` doubles after a 16-byte boundary, and the array around it."""
    import torch
    n = int(np.prod(shape))
    whole = torch.full((n + 8,), -7.0, dtype=torch.float64, pin_memory=pinned).numpy()
    at = 2 + skip + ((whole.ctypes.data >> 3) & 1)
    return whole[at:at + n].reshape(shape), whole, at


# 16, 96, 1920 and 10,080 sites end tiles of 32 or 16 sites; 73,728 sites are two chunks of the staged path
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 2), (6, 4, 10, 8), (10, 14, 6, 12), (18, 16, 16, 16)])
def test_links_get_buffers(dims, precision):
    import paper_0904_1179_gb300 as su3
    shape = su3.links_shape(dims)
    with su3.Lattice(dims, 5.7, 7, start=su3.SU3_HOT, precision=precision) as lat:
        want = lat.get_links()  # pageable
        np.testing.assert_allclose(np.einsum("...abx,...abx->...", want, want), 3.0, rtol=0, atol=1e-5)
        for pinned, skip in ((True, 0), (True, 1), (False, 0), (False, 1)):
            out, whole, at = _buffer(shape, pinned, skip)
            lat.get_links(out)
            assert out.tobytes() == want.tobytes()
            assert (whole[:at] == -7.0).all() and (whole[at + out.size:] == -7.0).all()
        if precision == 0:
            given = np.ascontiguousarray(want[..., ::-1, :, :, :])
            lat.set_links(given)
            out, _, _ = _buffer(shape, True, 0)
            assert lat.get_links(out).tobytes() == given.tobytes()


def test_batch_links_get_page_locked():
    import paper_0904_1179_gb300 as su3
    dims = [(4, 4, 4, 4), (6, 4, 2, 2), (8, 6, 4, 2)]
    with su3.Batch(dims, [5.7, 5.9, 6.1], [1, 2, 3], start=su3.SU3_HOT, precision=su3.SU3_FP32_MIXED) as b:
        b.sweep(2)
        for r, L in enumerate(dims):
            out, whole, at = _buffer(su3.links_shape(L), True, 0)
            assert b.get_links(r, out).tobytes() == b.get_links(r).tobytes()
            assert (whole[:at] == -7.0).all() and (whole[at + out.size:] == -7.0).all()
