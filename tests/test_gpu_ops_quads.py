"""The staggered-grid operators on four x-adjacent points per thread: buffers that start at an odd
float (scalar accesses) give bitwise the aligned (16-byte) result, at both block edges, on a set
with concave corners and single blocks, and equal the oracle's operators (1e-6 relative L2)."""
import numpy as np
import pytest

import oracle as O
from tests.helpers import built, rel_l2
from tests.rk_cases import from_blocks_dense, to_blocks_dense

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _odd(x):
    buf = torch.empty(x.numel() + 1, device="cuda")
    buf[1:] = x.reshape(-1)
    return buf[1:]


@pytest.mark.parametrize("B", [8, 16])
@pytest.mark.parametrize("op", [0, 1, 2, 3])
def test_alignment_and_edges(B, op):
    lgf = built()
    soln = np.array([[0, 0, 0], [1, 0, 0], [3, 1, 0], [0, 3, 2]], dtype=np.int32)
    dx = 0.25
    plan = lgf.RKPlan(B, soln, dx, 0.01, 100.0)
    xs = plan.blocks(0)
    rng = np.random.default_rng(B + op)
    nin, nout = (1 if op == 3 else 3), (1 if op == 2 else 3)
    origin = xs.min(0) - 1
    n = (xs.max(0) + 2 - origin)[::-1] * B
    f = rng.standard_normal((len(xs), nin, B, B, B)).astype(np.float32)
    x = torch.from_numpy(f).cuda()
    y = torch.empty((len(xs), nout, B, B, B), device="cuda")
    plan.op(op, x, y)
    z = _odd(torch.zeros_like(y))
    plan.op(op, _odd(x), z)
    assert torch.equal(y.reshape(-1), z)
    dense = from_blocks_dense(f.astype(np.float64), B, xs, origin, tuple(n))
    ref = {0: O.op_C, 1: O.op_Ct, 2: O.op_Gt, 3: O.op_G}[op](dense[0] if nin == 1 else dense, dx)
    ref = to_blocks_dense(ref[None] if ref.ndim == 3 else ref, B, xs, origin)
    assert rel_l2(y.cpu().numpy(), ref) < 1e-6
