"""The three-pass Poisson form where tests/test_gpu_plane.py does not go: 113 to 128 points on an axis
(the length 128), and planes that are long in y and z together, beyond the 2^18 points below which every
box takes the form.  Same parity bound, 1e-6 relative L2 against the FP64 oracle."""
import pytest

from tests.test_gpu_plane import _case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("e", [120, 128])
def test_length_128(axis, e):
    ext = [16, 16, 16]
    ext[axis] = e
    _case(ext, (0, 0, 0), (0, 0, 0), 1, odd=False)


# (x, y, z): planes of My x Mz between 64 x 128 and 80 x 256, three and four residues of y
@pytest.mark.parametrize("ext,ncomp", [((24, 96, 128), 3), ((32, 160, 144), 1), ((16, 104, 176), 2), ((24, 200, 192), 1),
                                       ((16, 160, 256), 1), ((40, 144, 208), 1), ((200, 136, 96), 1)])
def test_large_planes(ext, ncomp):
    _case(ext, (0, 0, 0), (0, 0, 0), ncomp, odd=False)


def test_large_plane_shifted():
    _case((24, 80, 120), (1, -2, -1), (0, 2, 1), 1, odd=True)
