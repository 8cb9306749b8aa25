"""The grey + downscale pass and the post-processing kernel against the oracle,
integer for integer (and float for float), where their groups and words end:
widths around the four-column groups, image bytes at every alignment, rows with
few or no matched pixels (the search for the nearest one crosses many mask
words), frames of both kinds in one batch."""
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


def _images(W, H, seed):
    rng = np.random.default_rng(seed)
    left = rng.integers(0, 256, (H, W, 3), dtype=np.uint8)
    right = rng.integers(0, 256, (H, W, 3), dtype=np.uint8)      # unrelated: matched pixels are rare
    right[H // 2:, : max(W - 6, 0)] = left[H // 2:, 6 if W > 6 else W:]   # the lower half matches
    return left, right


@pytest.mark.parametrize("downscale", [0, 1])
@pytest.mark.parametrize("W,H", [(2, 2), (3, 3), (5, 4), (6, 9), (7, 16), (130, 17), (131, 18), (132, 33), (133, 8),
                                 (700, 12), (1027, 10)])
def test_widths_alignments_and_sparse_matches(W, H, downscale):
    from paper_2212_00488_gb300 import Stereo, _lib
    left, right = _images(W, H, W * H)
    D = min(24, W)
    p = oracle.Params()
    p.downscale = downscale
    ref = oracle.pipeline(left, right, D, p)
    st = Stereo(0, downscale=downscale)
    for off in range(4):
        bufs = []
        for im in (left, right):
            b = torch.zeros(im.size + 8, dtype=torch.uint8, device="cuda")
            b[off:off + im.size] = torch.from_numpy(im.reshape(-1)).cuda()
            bufs.append(b)
        disp = torch.full((H, W), -1.0, device="cuda")
        X, Y = (W // 2, H // 2) if downscale else (W, H)
        gcp = torch.full((Y, X), 9, dtype=torch.uint8, device="cuda")
        _lib.stereo_compute(st.ctx, bufs[0].data_ptr() + off, bufs[1].data_ptr() + off, W, H, D, disp.data_ptr(),
                            0, 0, gcp.data_ptr())
        _lib.stereo_sync(st.ctx)
        planes = st.debug_planes(X, Y)
        torch.cuda.synchronize()
        assert np.array_equal(planes["grey_l"].cpu().numpy(), ref.grey_l)
        assert np.array_equal(planes["grey_r"].cpu().numpy(), ref.grey_r)
        assert np.array_equal(gcp.cpu().numpy(), ref.gcp)
        assert np.array_equal(disp.cpu().numpy(), ref.disp)
    st.close()


def test_batch_of_aligned_and_odd_frames():
    from paper_2212_00488_gb300 import Stereo, _lib
    sizes = [(64, 40), (65, 41), (66, 42), (67, 43), (68, 44), (130, 20)]
    for n in (len(sizes), 3):                 # through a graph, and directly
        frames, jobs = [], []
        for i, (W, H) in enumerate(sizes[:n]):
            left, right = _images(W, H, i)
            t = [torch.from_numpy(a).cuda() for a in (left, right)]
            disp = torch.full((H, W), -1.0, device="cuda")
            frames.append((left, right, t, disp))
            jobs.append(_lib.stereo_job(t[0].data_ptr(), t[1].data_ptr(), W, H, 20, disp.data_ptr(), None, None, None))
        st = Stereo(0)
        torch.cuda.synchronize()
        for _ in range(2):
            _lib.stereo_compute_batch(st.ctx, jobs)
            _lib.stereo_sync(st.ctx)
        for left, right, _, disp in frames:
            assert np.array_equal(disp.cpu().numpy(), oracle.pipeline(left, right, 20, oracle.Params()).disp)
        st.close()
