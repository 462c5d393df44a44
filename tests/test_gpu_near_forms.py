"""Which of the two quad forms near_form 3 takes, and the direct one's results: sheets, columns along x
and dense boxes have too few row-steps for what a tile stages and stay direct, with full quads, empty
slots and halves, and several quads per warp; compact sets with their neighbours go to the tiles.
Against the FP64 direct sum at the split method's bound, 1e-6 relative L2."""
import numpy as np
import pytest

from tests.helpers import built, oracle_poisson_blocks, rel_l2
from tests.test_gpu_near_tiles import _box
from tests.test_gpu_split import _dilate, _plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIRECT, TILES = 3, 4


@pytest.mark.parametrize("src_c,reach,ncomp,form", [
    (_box(24, 24, 1, (-9, -5, 2)), 0, 1, DIRECT),  # a sheet: full quads
    (_box(17, 1, 1, (-3, -1, -7)), 1, 2, DIRECT),  # a row and its neighbours: empty slots and halves
    (_box(8, 8, 8), 0, 1, DIRECT),                 # a dense box: 16 quads in a block's eight warps
    (_box(4, 4, 4, (-2, -2, -2)), 1, 1, TILES),
    (_box(8, 8, 1), 1, 1, TILES),                  # a sheet with its neighbours
])
def test_near_form(src_c, reach, ncomp, form):
    lgf = built()
    B = 16
    rng = np.random.default_rng(12)
    dst_c = _dilate(src_c, reach) if reach else src_c
    f = np.zeros((len(src_c), ncomp, B * B * B), dtype=np.float32)
    for b in range(len(src_c)):  # 12 random points per block keep the direct sum small
        for c in range(ncomp):
            f[b, c, rng.choice(B * B * B, 12, replace=False)] = rng.standard_normal(12)
    f = f.reshape(len(src_c), ncomp, B, B, B)
    _, plan = _plan(lgf, src_c, dst_c, ncomp=ncomp, scale=-1.0, dx=0.5, near_form=3)
    assert plan.near_form() == (form, [-1.0] * 4)
    d_dst = torch.full((len(dst_c), ncomp, B, B, B), 9.0, device="cuda")
    plan.execute([torch.from_numpy(f).cuda()], [d_dst])
    out = d_dst.cpu().numpy()
    K = lgf.required_max_offset(src_c, dst_c, B)
    pick = rng.integers(0, B, (len(dst_c), 6, 3))  # six points of every target block
    pts = (dst_c[:, None, :] * B + pick).reshape(-1, 3)
    for c in range(ncomp):
        got = out[np.arange(len(dst_c))[:, None], c, pick[..., 2], pick[..., 1], pick[..., 0]].reshape(-1)
        ref = oracle_poisson_blocks(f, src_c, B, pts, K, comp=c, scale=-1.0, dx=0.5)
        assert rel_l2(got, ref) < 1e-6, c
    plan.check()


def test_forms_timed_at_plan_time():
    lgf = built()
    _, plan = _plan(lgf, _box(3, 3, 3), _dilate(_box(3, 3, 3), 1))
    form, ms = plan.near_form()
    assert min(ms) > 0 and form == 1 + int(np.argmin(ms))
    t = lgf.Table(lgf.LAPLACE7, max_offset=31)
    assert lgf.Plan(t, [lgf.Solve(16, 1, _box(1, 1, 1), _box(1, 1, 1))]).near_form() == (0, [-1.0] * 4)
