"""The differentiable form on the GPU (FP32) against the FP64 oracle, where its
tiles, segments and spans end: images of a few pixels with many disparities.

Bounds come from FP32 rounding. An aggregated cost is a direct sum of at most
(2 wx + 1) + (2 wy + 1) positive rounded terms, with 32 rounding errors allowed for
expf, the grey values and the normalisation: a relative error of at most
rel = (2 wx + 2 wy + 34) 2^-24 (about 1e-5 at wx 21, wy 31). z = -CA / tau moves by
at most |z| rel, dhat by at most D max|z| rel, and a gradient, whose terms hold
p_d twice and sums of few hundred terms, by a small multiple of max|z| rel: 2e-3 of
the largest at rel = 1e-5, as in the tests of the other shapes. The images are
grey (R = G = B), so that two greys are equal in FP32 exactly where they are in
FP64 and the subgradient at the kink of Eq. 4 is the same; the incoming gradient
has one sign, so that the sums over pixels keep their size."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

THETA = [1.0, 1.0, 0.3, 2.3]
TAU = 0.1


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_00488_gb300 import build
    build.build()


def _grey_images(B, W, H, seed):
    """uint8 grey pairs of flat patches of many sizes (arms of every length up to
    the caps) with steps above the arm threshold between them, noise of 0 to 4."""
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(2 * B):
        im = np.full((H, W), 60)
        for _ in range(6):
            x0, y0 = rng.integers(0, W), rng.integers(0, H)
            im[y0:y0 + rng.integers(1, H + 1), x0:x0 + rng.integers(1, W + 1)] = rng.choice((60, 90, 120, 150))
        out.append((im + rng.integers(0, 5, (H, W))).astype(np.uint8))
    rgb = np.repeat(np.stack(out)[..., None], 3, axis=3)
    return np.ascontiguousarray(rgb[:B]), np.ascontiguousarray(rgb[B:]), rng.uniform(0.5, 1.5, (B, H, W))


def _step(lu, ru, go, D, wx, wy):
    from paper_2212_00488_gb300 import Stereo
    from paper_2212_00488_gb300.diff import soft_argmin_disparity
    st = Stereo(0, downscale=0, wx=wx, wy=wy, cost_scale=9)   # (not used here; lets wx reach its limit)
    l, r = (torch.from_numpy(a.astype(np.float32) / 255).cuda().requires_grad_(True) for a in (lu, ru))
    theta = torch.tensor(THETA, device="cuda", requires_grad=True)
    dhat = soft_argmin_disparity(l, r, theta, torch.from_numpy(lu).cuda(), torch.from_numpy(ru).cuda(), D, TAU, st)
    grads = torch.autograd.grad(dhat, (l, r, theta), torch.from_numpy(go.astype(np.float32)).cuda())
    res = [t.detach().cpu().numpy().astype(np.float64) for t in (dhat, *grads)]
    st.close()
    return res


def _check(B, W, H, D, wx, wy, seed=0):
    lu, ru, go = _grey_images(B, W, H, 1000 * W + H + seed)
    go = go.astype(np.float32)
    dhat, gl, gr, gt = _step(lu, ru, go, D, wx, wy)
    rel = (2 * wx + 2 * wy + 34) * 2.0 ** -24
    tol = 2e-3 * max(1.0, rel / 1e-5)
    red = 77.0 / 256.0
    theta_sum = np.zeros(4)
    for b in range(B):
        q = [oracle.grey(im[b]) for im in (lu, ru)]
        g = [oracle.grey_f((im[b].astype(np.float32) / 255).astype(np.float64)) for im in (lu, ru)]
        want, wl, wr, wt = oracle.diff_forward_backward(
            g[0], g[1], oracle.census(q[0]), oracle.census(q[1]), oracle.arms(q[0], wx, wy, 13), D,
            np.array(THETA), tau=TAU, go=go[b].astype(np.float64))
        theta_sum += wt
        assert np.abs(dhat[b] - want).max() <= D * (2.0 / TAU) * rel, b
        for got, exp in ((gl[b, ..., 0] / red, wl), (gr[b, ..., 0] / red, wr)):
            assert np.linalg.norm(got - exp) <= tol * np.linalg.norm(exp), b
            assert np.abs(got - exp).max() <= tol * np.abs(exp).max(), b
    assert np.allclose(gt, theta_sum, rtol=tol, atol=1e-4 * np.abs(theta_sum).max()), (gt, theta_sum)


# few pixels, many chunks of disparities: more partials of the parameter gradients than pixels
@pytest.mark.parametrize("B,W,H,D,wy", [(64, 1, 1, 256, 31), (4, 1, 1, 256, 31), (16, 1, 12, 256, 31),
                                        (3, 4, 4, 256, 0), (8, 3, 8, 256, 0), (2, 2, 70, 256, 31)])
def test_images_of_a_few_pixels(B, W, H, D, wy):
    _check(B, W, H, D, 21, wy)


# 142 bytes a pixel and pair, and the partials (16 bytes for two rows of a segment
# and chunk, fewer in narrow images): capped contexts run the step
@pytest.mark.parametrize("B,W,H,D,cap_per_pixel", [(2, 300, 200, 24, 150), (1, 2, 4000, 256, 200)])
def test_workspace_holds_only_planes_in_use(B, W, H, D, cap_per_pixel):
    from paper_2212_00488_gb300 import Stereo, _lib
    from paper_2212_00488_gb300.diff import soft_argmin_disparity
    lu, ru, go = _grey_images(B, W, H, 3)
    res = []
    for cap in (0, cap_per_pixel * B * W * H):
        st = Stereo(0, downscale=0, mem_cap_bytes=cap)
        l, r = (torch.from_numpy(a.astype(np.float32) / 255).cuda().requires_grad_(True) for a in (lu, ru))
        theta = torch.tensor(THETA, device="cuda", requires_grad=True)
        dhat = soft_argmin_disparity(l, r, theta, torch.from_numpy(lu).cuda(), torch.from_numpy(ru).cuda(), D, TAU, st)
        res.append((dhat.detach(), *torch.autograd.grad(dhat.sum(), (l, r, theta))))
        torch.cuda.synchronize()
        st.close()
    for a, b in zip(*res):
        assert torch.equal(a, b)
    st = Stereo(0, downscale=0, mem_cap_bytes=100 * B * W * H)
    with pytest.raises(_lib.StereoError) as e:
        soft_argmin_disparity(*(torch.from_numpy(a.astype(np.float32)).cuda() for a in (lu, ru)),
                              torch.tensor(THETA, device="cuda"), torch.from_numpy(lu).cuda(),
                              torch.from_numpy(ru).cuda(), D, TAU, st)
    assert e.value.code == _lib.STEREO_ENOMEM
    st.close()


# windows of one row or one column, spans past 32 cells, arms at every cap, wide
# windows, one pair more than a support launch takes, segments' and bands' edges,
# more disparities than columns
@pytest.mark.parametrize("B,W,H,D,wx,wy", [(1, 70, 40, 12, 0, 0), (2, 65, 33, 9, 21, 0), (1, 40, 70, 9, 0, 31),
                                           (1, 120, 90, 20, 21, 31), (1, 90, 70, 8, 5, 5), (1, 300, 80, 12, 141, 31),
                                           (1, 261, 67, 17, 61, 15), (33, 31, 9, 5, 21, 31), (1, 1100, 9, 24, 21, 31),
                                           (1, 505, 6, 8, 21, 31), (1, 506, 6, 9, 21, 31), (1, 3, 40, 16, 21, 31),
                                           (1, 20, 12, 64, 21, 31)])
def test_windows_segments_and_batches(B, W, H, D, wx, wy):
    _check(B, W, H, D, wx, wy)


def test_overflowing_parameter_gradient_stays_infinite():
    # Windows of one pixel, two disparities: the left image is the right one, its
    # columns take two greys in turn, so only the cells of disparity 1 have a cost and
    # every pixel's share of d/d w_AD and d/d w_MC is about -1.8e38, of d/d lambda_AD
    # 1e37: the sums pass the largest float in one direction.
    from paper_2212_00488_gb300 import Stereo
    from paper_2212_00488_gb300.diff import soft_argmin_disparity
    W, H = 400, 4
    im = np.where(np.arange(W) % 2 == 0, 51, 153).astype(np.uint8)
    im = np.ascontiguousarray(np.broadcast_to(im[None, None, :, None], (1, H, W, 3)))
    u = torch.from_numpy(im).cuda()
    f = u.float() / 255
    theta = torch.tensor([0.05, 0.0, 0.3, 2.3], device="cuda", requires_grad=True)
    st = Stereo(0, downscale=0, wx=0, wy=0)
    dhat = soft_argmin_disparity(f, f.clone(), theta, u, u.clone(), 2, 0.1, st)
    gt, = torch.autograd.grad(dhat, (theta,), torch.full((1, H, W), 1e38, device="cuda"))
    st.close()
    inf = float("inf")
    assert gt[:3].tolist() == [-inf, -inf, inf]
