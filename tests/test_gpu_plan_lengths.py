"""Plan.lengths: the form and the padded lengths that a plan runs, for both whole-box forms, an autotuned
and a split plan, and bad arguments."""
import numpy as np
import pytest

from paper_1601_00035_gb300 import inputs
from tests.helpers import built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_lengths():
    lgf = built()
    c = inputs.block_grid((48, 32, 96), 16).astype(np.int32)  # z, y, x
    t = lgf.Table(lgf.LAPLACE7, max_offset=lgf.required_max_offset(c, c, 16))
    solve = lgf.Solve(16, 1, c, c)
    p = lgf.Plan(t, [solve, solve])
    passes, n = p.lengths(1)
    assert passes == 3 and n[0] == 192 and n[2] == 96 and 64 <= n[1] <= 96
    assert p.lengths(2)[0] == p.lengths(-1)[0] == -1
    # five passes on the lengths of the size rule
    assert lgf.Plan(t, [solve], precision=1).lengths() == (5, [lgf.fft_length(2 * e) for e in (96, 32, 48)])
    assert lgf.Plan(t, [solve], method=1).lengths() == (0, [0, 0, 0])
    q = lgf.Plan(t, [solve], method=2)
    assert q.lengths() == ((0, [0, 0, 0]) if q.method()[0] == 1 else (passes, n))
