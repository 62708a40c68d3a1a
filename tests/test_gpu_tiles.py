"""Calls that tile_detect_kernel takes (small and middling ones) give the bytes of the oracle and of the
persistent kernels, whatever form takes them."""
import numpy as np
import pytest

import oracle
from paper_2003_13493_gb300 import synth, vio

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def on_gpu(img, pad=0, offset=0):
    h, w = img.shape
    pitch = w + pad
    buf = torch.full((h * pitch + offset + 64,), 255, dtype=torch.uint8, device="cuda")
    v = buf[offset:offset + h * pitch].view(h, pitch)[:, :w]
    v.copy_(torch.from_numpy(img))
    return v


def check(sizes, levels, arc=9, thresh=12, cell=32, score=0, radius=1, pad16=True, pyramid=False):
    imgs = [synth.make_frame(w, h, seed=w * 7 + h + i) for i, (w, h) in enumerate(sizes)]
    frames = [on_gpu(im, (-im.shape[1]) % 16 if pad16 else 3) for im in imgs]
    det = vio.Detector(max_frames=len(sizes), score=score, nms_radius=radius)
    for _ in range(2):  # the second call finds keys and counters cleared by the first
        outs, counts = det.detect(frames, thresh, arc, cell, levels)
    det.sync()
    got = [o.cpu().numpy() for o in outs], counts.cpu().numpy()
    if pyramid:
        for i, im in enumerate(imgs):
            for k, want in enumerate(oracle.pyramid(im, levels)):
                assert np.array_equal(det.copy_level(i, k), want), (sizes[i], k)
    det.set_variant(vio.variant_ids(radius)[0])  # a pinned variant takes the persistent kernels
    outs, counts = det.detect(frames, thresh, arc, cell, levels)
    det.sync()
    for i, im in enumerate(imgs):
        assert np.array_equal(got[0][i], outs[i].cpu().numpy()), sizes[i]
        want, n = oracle.detect(im, thresh, arc, cell, levels, score, nms_radius=radius)
        assert np.array_equal(got[0][i], want) and got[1][i] == n == int(counts[i]), sizes[i]
    det.close()


EDGES = [(7, 7), (16, 30), (31, 33), (119, 61), (120, 62), (121, 63), (128, 64), (240, 124), (249, 126), (368, 187)]


# up to 8 frames: 30-row tiles in one launch; more: 62-row tiles in one launch
@pytest.mark.parametrize("n", [1, 8, 10])
def test_one_level(n):
    check(EDGES[-n:] if n > 1 else [(121, 63)], 1)


@pytest.mark.parametrize("n", [5, 9])
@pytest.mark.parametrize("levels", [2, 3])
def test_one_launch_builds_the_pyramid(n, levels):
    check([(28, 28), (120, 62), (121, 125), (361, 129), (752, 480), (480, 97), (240, 248), (129, 253), (97, 60)][:n],
          levels, pyramid=True)


@pytest.mark.parametrize("levels", [1, 2, 3])
def test_one_launch_and_a_decode_launch(levels):
    """More than 800 tiles of 62 rows."""
    check([(1920, 1080), (1921, 1083), (361, 129), (2000, 1100)], levels)


@pytest.mark.parametrize("levels", [4, 5])
@pytest.mark.parametrize("pad16", [True, False])
def test_two_launches(levels, pad16):
    check([(112, 112), (120, 124), (121, 187), (497, 255), (752, 480), (963, 248)], levels, pad16=pad16, pyramid=True)


@pytest.mark.parametrize("radius", [1, 2, 3, 4])
@pytest.mark.parametrize("score", [0, 1, 2])
def test_radius_and_score(radius, score):
    check([(368, 187), (121, 70)], 3, score=score, radius=radius, arc=10)
    check([(368, 187)] * 3, 4, score=score, radius=radius, cell=64)


@pytest.mark.parametrize("thresh,arc", [(0, 9), (1, 16), (127, 9), (128, 9), (200, 12), (255, 10)])
def test_thresholds_and_arcs(thresh, arc):
    check([(368, 187)], 3, thresh=thresh, arc=arc)


def test_dense_corners_and_streams():
    """Noise at a low threshold fills the queues; calls that alternate streams and forms keep their order."""
    rng = np.random.default_rng(4)
    imgs = [rng.integers(0, 256, (187, 368)).astype(np.uint8) for _ in range(12)]
    want = [oracle.detect(im, 2, 9, 32, 3) for im in imgs]
    det = vio.Detector(max_frames=16)
    frames = [on_gpu(im) for im in imgs]
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    got = []
    for r in range(12):
        n = (1, 12, 3)[r % 3]
        with torch.cuda.stream(streams[r % 2]):
            got.append((n, det.detect(frames[:n], 2, 9, 32, 3, stream=streams[r % 2])))
    for s in streams:
        det.sync(s)
    for n, (outs, counts) in got:
        for i in range(n):
            assert np.array_equal(outs[i].cpu().numpy(), want[i][0]) and int(counts[i]) == want[i][1]
    det.close()
