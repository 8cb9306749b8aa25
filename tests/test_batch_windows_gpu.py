"""Batches whose windows take the split packed tiles (W_x 41 and 61), and batches
without downscaling, against the oracle, integer for integer and float for float:
several tiles and bands for each CTA of the persistent kernel, frames of odd
sizes, directly and through a graph."""
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


def _check(sizes, downscale, tile, **params):
    from paper_2212_00488_gb300 import Stereo, _lib
    frames, jobs = [], []
    for i, (W, H, D) in enumerate(sizes):
        s = scenes.make_scene(W, H, D, planes=5, seed=W + i)
        left, right = s.left // 64 + 100, s.right // 64 + 100          # arms at their caps
        X, Y = (W // 2, H // 2) if downscale else (W, H)
        t = [torch.from_numpy(a).cuda() for a in (left, right)]
        o = [torch.full((H, W), -1.0, device="cuda")] + [torch.full((Y, X), 99, dtype=torch.uint8, device="cuda")
                                                        for _ in range(3)]
        frames.append((left, right, D, t, o))
        jobs.append(_lib.stereo_job(t[0].data_ptr(), t[1].data_ptr(), W, H, D, *(q.data_ptr() for q in o)))
    st = Stereo(0, downscale=downscale, **params)
    _lib.stereo_set_tile(st.ctx, tile)
    torch.cuda.synchronize()
    for _ in range(2):
        _lib.stereo_compute_batch(st.ctx, jobs)
        _lib.stereo_sync(st.ctx)
    st.close()
    p = oracle.Params()
    p.downscale = downscale
    for k, v in params.items():
        setattr(p, k, v)
    for left, right, D, _, o in frames:
        ref = oracle.pipeline(left, right, D, p)
        for got, want in zip(o, (ref.disp, ref.dl, ref.dr, ref.gcp)):
            assert np.array_equal(got.cpu().numpy(), want), (left.shape, D)


SIZES = [(300, 150, 40), (131, 97, 21), (200, 61, 9), (97, 64, 30), (64, 33, 5)]


@pytest.mark.parametrize("n", [2, 5])
@pytest.mark.parametrize("wx,tile", [(41, 3), (41, 8), (61, 8), (61, -1)])
def test_split_tiles_in_a_batch(wx, tile, n):
    _check(SIZES[:n], 0, tile, wx=wx, wy=15)


# more tiles than SMs: every CTA of the persistent kernel takes several
@pytest.mark.parametrize("wx,tile", [(21, -1), (61, 8)])
def test_several_tiles_a_cta(wx, tile):
    _check([(700, 90, 60)] * 3, 0, tile, wx=wx, wy=15)


@pytest.mark.parametrize("n", [2, 5])
def test_split_tiles_with_downscaling(n):
    _check([(2 * W, 2 * H, 2 * D) for W, H, D in SIZES[:n]], 1, 8, wx=61, wy=15)
