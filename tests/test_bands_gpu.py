"""Row bands and slab edges of the fused kernel against the oracle, integer for
integer: frames tall and narrow enough to be cut into bands, arms at the caps so
that windows cross every band border, strips one column either side of a tile's
width, and disparity counts that make the last slab overlap the one before it
(or fall short of one slab)."""
import numpy as np
import pytest

import oracle
from paper_2212_00488_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_00488_gb300 import build
    build.build()


@pytest.mark.parametrize("tile", [-1, 0, 3, 4, 5, 8])
@pytest.mark.parametrize("W,H,D", [(40, 901, 9), (95, 130, 3), (96, 61, 4), (97, 300, 5), (193, 257, 75)])
def test_bands_and_overlapping_slabs(W, H, D, tile):
    _check(W, H, D, tile)


# more tiles than one wave: whole tiles first, the rest in bands
@pytest.mark.parametrize("tile", [-1, 0, 1, 2, 3, 4, 5, 6, 7, 8])
def test_whole_tiles_and_banded_rest(tile):
    _check(1000, 130, 75, tile)


# windows above 2^16 that the split form of tiles 3 and 8 takes (wx 41 and 61 at
# scale 512, and at the last scale it takes), and the 32-bit form just past it
@pytest.mark.parametrize("tile,wx,scale", [(3, 41, 512), (8, 61, 512), (-1, 58, 512), (3, 58, 587), (3, 58, 588),
                                           (8, 66, 517), (8, 66, 518), (-1, 41, 1300)])
def test_windows_above_16_bits(tile, wx, scale):
    _check(300, 90, 18, tile, wx=wx, wy=15, cost_scale=scale)


def _check(W, H, D, tile, **params):
    from paper_2212_00488_gb300 import Stereo, _lib
    s = scenes.make_scene(W, H, D, planes=5, seed=W + H)
    left, right = s.left // 64 + 100, s.right // 64 + 100          # arms at their caps
    st = Stereo(0, downscale=0, **params)
    _lib.stereo_set_tile(st.ctx, tile)
    out = st(torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda(), D, maps=True)
    torch.cuda.synchronize()
    st.close()
    p = oracle.Params()
    p.downscale = 0
    for k, v in params.items():
        setattr(p, k, v)
    ref = oracle.pipeline(left, right, D, p)
    for k in ("dl", "dr", "gcp", "disp"):
        got, want = getattr(out, k).cpu().numpy(), getattr(ref, k)
        bad = np.argwhere(got != want)
        assert bad.size == 0, f"{k}: {len(bad)} mismatches, first {bad[:5].tolist()}"
