"""The support kernel (mini-census codes and cross arms) against the oracle,
integer for integer, at the edges of its 128 x 16 pixel tiles, of its four-pixel
words and of its byte compare (tc on both sides of 128), with arms of every
length up to the caps, with few CTAs (two on an SM) and with more (three)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_00488_gb300 import build
    build.build()


@pytest.mark.parametrize("W,H", [(1, 1), (3, 9), (4, 5), (5, 3), (127, 15), (128, 16), (129, 17), (390, 70),
                                 (1217, 255)])
@pytest.mark.parametrize("tc,wx,wy", [(0, 21, 31), (13, 1, 1), (13, 6, 30), (127, 21, 31), (128, 21, 31),
                                      (255, 141, 31), (256, 5, 3)])
def test_codes_and_arms_at_tile_edges(W, H, tc, wx, wy):
    from paper_2212_00488_gb300 import Stereo
    rng = np.random.default_rng(W * 1000 + H)
    # steps of 0 to 2 levels along both axes, with full-range jumps here and there
    img = rng.integers(0, 3, (2, H, W)).cumsum(1).cumsum(2) + 255 * (rng.random((2, H, W)) < 0.02)
    rgb = np.repeat((img % 256).astype(np.uint8)[..., None], 3, axis=3)
    st = Stereo(0, downscale=0, wx=wx, wy=wy, tc=tc, cost_scale=9)
    left, right = (torch.from_numpy(np.ascontiguousarray(i)).cuda() for i in rgb)
    st(left, right, 4)
    got = st.debug_planes(W, H)
    torch.cuda.synchronize()
    for side, im in zip("lr", rgb):
        g = oracle.grey(im)
        arms = np.stack(oracle.arms(g, wx, wy, tc)).astype(np.int64)
        want = arms[0] | arms[1] << 8 | arms[2] << 16 | arms[3] << 24
        assert np.array_equal(got["census_" + side].cpu().numpy(), oracle.census(g))
        assert np.array_equal(got["arms_" + side].cpu().numpy().view(np.uint32).astype(np.int64), want)
    st.close()


# either side of the line up to which CTAs of eight rows each have an SM (150 and
# 156 of them on 152 SMs), and with fewer than four columns
@pytest.mark.parametrize("W,H", [(300, 200), (300, 208), (2, 30)])
@pytest.mark.parametrize("tc,wx,wy", [(13, 21, 31), (200, 141, 31), (40, 61, 7), (13, 0, 0)])
def test_rows_of_a_cta(W, H, tc, wx, wy):
    test_codes_and_arms_at_tile_edges(W, H, tc, wx, wy)
