"""The near-field multiply-accumulate on quads of targets, in tiles and direct (near_form 3), at the
edges of the tiles: a single tile, several, quads with empty slots and halves, negative block
coordinates, two components, and a dense box whose tiles hold few quads (the direct form).  Against
the FP64 direct sum at the split method's bound, 1e-6 relative L2."""
import numpy as np
import pytest

from tests.helpers import built, oracle_poisson_blocks, rel_l2
from tests.test_gpu_split import _dilate, _plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _box(nx, ny, nz, org=(0, 0, 0)):
    return np.array([[x + org[0], y + org[1], z + org[2]] for z in range(nz) for y in range(ny) for x in range(nx)],
                    dtype=np.int32)


def _scattered():
    return np.unique(np.random.default_rng(5).integers(-6, 6, (60, 3)).astype(np.int32), axis=0)


@pytest.mark.parametrize("src_c,reach,ncomp", [
    (_box(1, 1, 1), 0, 1),               # one target: direct, one slot of eight
    (_box(2, 2, 2, (-1, 3, -5)), 1, 2),  # 24 quads in one tile
    (_box(1, 1, 12, (-3, -1, -7)), 2, 1),  # a column: half-empty quads, several tiles
    (_scattered(), 1, 2),                # many tiles, most source slots absent
    (_box(7, 6, 5), 0, 1),               # dense: few quads to a tile
])
def test_near_tiles(src_c, reach, ncomp):
    lgf = built()
    B = 16
    rng = np.random.default_rng(11)
    dst_c = _dilate(src_c, reach) if reach else src_c
    f = np.zeros((len(src_c), ncomp, B * B * B), dtype=np.float32)
    for b in range(len(src_c)):  # 12 random points per block keep the direct sum small
        for c in range(ncomp):
            f[b, c, rng.choice(B * B * B, 12, replace=False)] = rng.standard_normal(12)
    f = f.reshape(len(src_c), ncomp, B, B, B)
    _, plan = _plan(lgf, src_c, dst_c, ncomp=ncomp, scale=-1.0, dx=0.5, near_form=3)
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
