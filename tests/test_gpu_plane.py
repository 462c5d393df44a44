"""GPU parity of the three-pass Poisson form (FP32 plans up to 512-point axes) at the edges of
its transform lengths, on each axis: every multiple of 16 a plane can have, y extents that
fold into several residues, targets shifted both ways (wrapped positions), and buffers that
start at an odd float.  Against the oracle's FP64 FFT convolution at the FP32 target of 1e-6
relative L2, on white-noise sources over a holed block set.
"""
import numpy as np
import pytest

import oracle as O
from paper_1601_00035_gb300 import inputs
from tests.helpers import built, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(ext, shift, grow, ncomp, odd, graph=False, B=8):
    """Sources on the blocks of a box of `ext` cells (every corner block present, a third of the
    others missing), targets on a box `grow` blocks wider, moved by `shift` blocks."""
    lgf = built()
    rng = np.random.default_rng(sum(ext) + 7 * sum(shift))
    box = inputs.block_grid(tuple(ext[::-1]), B)
    hi = box.max(0)
    src = box[(rng.random(len(box)) < 0.67) | (box == 0).all(1) | (box == hi).all(1)]
    tgt = inputs.block_grid(tuple((np.array(ext) + np.array(grow) * B)[::-1]), B) + np.array(shift, dtype=np.int32)
    tgt = tgt.astype(np.int32)
    f = rng.standard_normal((len(src), ncomp, B, B, B)).astype(np.float32)
    n = len(tgt) * ncomp * B ** 3
    pad = 1 if odd else 0
    src_buf, dst_buf = torch.zeros(f.size + pad, device="cuda"), torch.zeros(n + pad, device="cuda")
    s, d = src_buf[pad:], dst_buf[pad:]
    s.copy_(torch.from_numpy(f.reshape(-1)))
    t = lgf.Table(lgf.LAPLACE7, max_offset=lgf.required_max_offset(src, tgt, B))
    plan = lgf.Plan(t, [lgf.Solve(B, ncomp, src, tgt, dx=0.5, scale=-1.0)], use_graph=graph)
    plan.execute([s], [d])
    torch.cuda.synchronize()
    plan.set_profiling(2)
    again = torch.empty_like(dst_buf)[pad:]
    plan.execute([s], [again])
    torch.cuda.synchronize()
    assert "yz_conv" in plan.kernel_times()          # the form under test ran
    assert torch.equal(again, d)
    got = d.cpu().numpy().reshape(len(tgt), ncomp, B, B, B)
    dense = inputs.from_blocks(f.astype(np.float64), B, src, tuple(ext[::-1]))
    shape = tuple((np.array(ext) + np.array(grow) * B)[::-1])
    ref = -0.25 * O.fft_conv(dense, (0, 0, 0), tuple(np.array(shift) * B), shape)
    out = inputs.from_blocks(got, B, tgt - np.array(shift), shape)
    for c in range(ncomp):
        assert rel_l2(out[c], ref[c]) < 1e-6, (c, rel_l2(out[c], ref[c]))


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("e", [8, 24, 40, 56, 72, 88, 104, 136, 152, 168, 184, 200, 216, 232, 256])
def test_lengths(axis, e):
    ext = [16, 16, 16]
    ext[axis] = e
    _case(ext, (0, 0, 0), (0, 0, 0), 1, odd=False)


@pytest.mark.parametrize("ext,shift,grow", [((40, 24, 48), (-1, -1, -1), (2, 2, 2)), ((24, 56, 32), (1, 0, 2), (0, 1, 0)),
                                            ((80, 72, 88), (0, 2, -2), (1, 0, 2)), ((16, 200, 24), (0, -3, 0), (0, 6, 0)),
                                            ((104, 16, 136), (-2, 0, 1), (2, 1, 0)), ((112, 120, 96), (0, -1, -1), (1, 2, 2))])
@pytest.mark.parametrize("ncomp,odd,graph", [(1, False, True), (3, True, False), (2, False, False)])
def test_shifted_targets(ext, shift, grow, ncomp, odd, graph):
    _case(ext, shift, grow, ncomp, odd, graph)
