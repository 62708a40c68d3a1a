"""Frames that TMA cannot address (any base address or pitch): the pyramid
kernel copies them as it reads them, in detection, sweep and tracking."""
import numpy as np
import pytest

from paper_2003_13493_gb300 import synth, vio


def test_chunk_rows_and_columns():
    """Chunk number -> (row, column) with one multiply-high, corrected for a block's
    first chunk, exact for its threads: every chunk of a frame once."""
    rng = np.random.default_rng(3)
    for w in [7, 16, 17, 33, 480, 752, 1021, 3840, 65535] + [int(x) for x in rng.integers(7, 65536, 40)]:
        cx = max(2, -(-w // 16))
        magic = -(-(1 << 32) // cx)
        rows = max(1, (1 << 28) // w // 2 + 1)
        n = cx * rows
        first = np.unique(np.concatenate([np.arange(0, min(n, 1 << 20), 256), n - 1 - np.arange(0, min(n, 1 << 16), 256)]))
        first = first[first >= 0].astype(np.uint64) // np.uint64(256) * np.uint64(256)
        row = ((first * np.uint64(magic)) >> np.uint64(32)).astype(np.int64)
        f = first.astype(np.int64)
        row -= row * cx > f
        assert np.array_equal(row, f // cx)
        off = np.arange(cx + 256, dtype=np.uint64)
        assert np.array_equal((off * np.uint64(magic)) >> np.uint64(32), off // np.uint64(cx))


def place(torch, img, offset, pitch):
    h, w = img.shape
    buf = torch.full((h * pitch + offset + 3,), 255, dtype=torch.uint8, device="cuda")
    v = buf[offset:offset + h * pitch].view(h, pitch)[:, :w]
    v.copy_(torch.from_numpy(img))
    return v


LAYOUTS = [(0, 0), (1, 0), (2, 5), (3, 16), (16, 1), (7, 9), (0, 12)]


@pytest.mark.gpu
@pytest.mark.parametrize("levels", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("size", [(113, 117), (160, 121), (257, 130), (1021, 765)])
def test_detection_of_unaligned_frames(levels, size):
    import oracle
    torch = pytest.importorskip("torch")
    det = vio.Detector(max_frames=16)
    w, h = size
    imgs = [synth.make_frame(w, h, seed=11 + i) for i in range(len(LAYOUTS))]
    frames = [place(torch, im, o, w + p) for im, (o, p) in zip(imgs, LAYOUTS)]
    outs, counts = det.detect(frames, 12, 9, 32, levels)
    sweep, scounts = det.detect_sweep(frames, [(8, 9), (20, 12)], 32, levels)
    det.sync()
    for i, im in enumerate(imgs):
        want, n = oracle.detect(im, 12, 9, 32, levels)
        assert np.array_equal(outs[i].cpu().numpy(), want) and int(counts[i]) == n, LAYOUTS[i]
        for p, (t, a) in enumerate([(8, 9), (20, 12)]):
            want, n = oracle.detect(im, t, a, 32, levels)
            assert np.array_equal(sweep[p][i].cpu().numpy(), want) and int(scounts[p, i]) == n, LAYOUTS[i]
    # level 0 reads back the frame's pixels
    outs, counts = det.detect(frames, 12, 9, 32, levels)
    for i, im in enumerate(imgs):
        for k, want in enumerate(oracle.pyramid(im, levels)):
            assert np.array_equal(det.copy_level(i, k), want), (i, k)
    det.close()


@pytest.mark.gpu
@pytest.mark.parametrize("levels", [1, 3])
def test_tracking_of_unaligned_pairs(levels):
    torch = pytest.importorskip("torch")
    det = vio.Detector(max_frames=4)
    w, h = 331, 243
    a, b = synth.smooth_frame(w, h, 5), synth.smooth_frame(w, h, 5, dx=1.5, dy=-0.75)
    pts = torch.tensor([[x, y] for y in range(40, 200, 20) for x in range(40, 290, 20)], dtype=torch.float32).cuda()
    got = []
    for offset, pad in ((0, 5), (0, 0), (3, 1)):
        pair = [place(torch, im, offset, w + pad) for im in (a, b)]
        got.append(det.track([pair[0]], [pair[1]], [pts], dict(levels=levels))[0].cpu().numpy())
    assert all(np.array_equal(g.view(np.int32), got[0].view(np.int32)) for g in got)
    assert (got[0].view(np.int32)[:, 4] == 1).mean() > 0.9
    det.close()


@pytest.mark.gpu
@pytest.mark.parametrize("size", [(40, 31), (23, 300), (300, 24), (33, 26), (96, 64)])
def test_tracking_near_borders_and_in_small_images(size):
    """Features everywhere, also where the pixel windows reach the border or the image is smaller than
    one: status as the oracle's, positions of the tracked ones (fixed iterations)."""
    torch = pytest.importorskip("torch")
    from oracle import lk_oracle as lk
    w, h = size
    a, b = synth.smooth_frame(w, h, 8), synth.smooth_frame(w, h, 8, dx=0.75, dy=-0.5)
    pts = np.array([[x, y] for y in np.arange(2.25, h - 2, 3.5) for x in np.arange(2.5, w - 2, 3.25)], np.float32)
    det = vio.Detector(max_frames=2)
    for levels in (1, 2) if min(w, h) >= 16 else (1,):
        p = dict(patch_fine=8, patch_coarse=8, max_iters=6, min_update=0.0, model=0)
        got = det.track([place(torch, a, 0, w + (-w) % 16)], [place(torch, b, 0, w + (-w) % 16)],
                        [torch.from_numpy(pts).cuda()], dict(p, levels=levels))[0].cpu().numpy()
        want = lk.track(a, b, pts.astype(np.float64), levels=levels, **p)
        status = got.view(np.int32)[:, 4]
        # a position that fp32 rounds across a border may flip a track near it
        assert (status != want[:, 4].astype(np.int32)).mean() <= 0.01
        more = lk.track(a, b, pts.astype(np.float64), levels=levels, **dict(p, max_iters=7))
        ok = (status == 1) & (want[:, 4] == 1) & (np.abs(want[:, :2] - more[:, :2]).max(axis=1) < 1e-6)
        # (on two levels every patch of the narrow images leaves the coarse one)
        assert (ok.sum() > 0 or levels == 2) and np.abs(got[ok, :2] - want[ok, :2]).max(initial=0) < 1e-3
    det.close()
