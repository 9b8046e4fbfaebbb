"""fd_forward_noalloc's size limit, checked before any device call: a y-z plane of
more than 16,384 tiles of 8 x 32 points is refused and the error names that limit (the
kernel's scratch is one word: nothing else bounds the plane); a plane of exactly that
many is not refused for its size (no step is asked for, so no buffer is touched)."""
import pytest

import paper_1912_00695_gb300 as fd
from paper_1912_00695_gb300 import _abi


def _call(ny, nz):
    _abi.fd_forward_noalloc(64, 64, 64, None, (4, ny, nz), 8, 10.0, 1e-3, nt=0, want_amax=False)


@pytest.mark.parametrize("ny,nz", [(4200, 4200), (16385, 256), (65535, 65)])
def test_too_large_a_plane_is_refused(ny, nz):
    with pytest.raises(fd.FdError) as e:
        _call(ny, nz)
    assert e.value.code == fd.FD_EINVAL
    assert "16384 tiles of 8 x 32 points" in fd.fd_last_error()
    assert "scratch" not in fd.fd_last_error()


@pytest.mark.parametrize("ny,nz", [(16384, 256), (65535, 64), (8, 65535)])
def test_the_largest_planes_are_taken(ny, nz):
    try:
        _call(ny, nz)
    except fd.FdError as e:  # (a machine without a GPU)
        assert e.code != fd.FD_EINVAL
