"""bench.py's model of the three-pass form: the yz pass on the lengths that the plan runs (224 x 256 x
256 for the 128^3 ring), its own spectrum array (all of y) and the transforms it does, worked out here
from the shapes."""
import math

import numpy as np


def test_yz_pass_model():
    import bench
    B = bench.B
    src = np.array([[1, 1, 1], [6, 5, 4]])
    dst = np.array([[0, 0, 0], [7, 7, 7]])
    N = [224, 256, 256]
    g = bench.geometry(src, dst, 3, N)
    assert (g["Es"], g["Et"], g["N"]) == ([6 * B, 5 * B, 4 * B], [8 * B] * 3, N)
    kx = 113  # real rows of 224
    line = 5.0 * 256 * math.log2(256)
    y = kx * (4 * B + 8 * B) * line           # rows along y: forward on the source's z, inverse on the target's
    z = kx * 256 * (2 * line + 2 * 256)       # columns along z: there, times the spectrum, and back
    assert math.isclose(bench.pass_flops(g)["yz_conv"], 3 * (y + z))
    arrays = 3 * 8 * kx * (4 * B * 5 * B + 8 * B * 8 * B)
    assert bench.pass_bytes(g)["yz_conv"] == arrays + 4 * kx * 256 * 129
