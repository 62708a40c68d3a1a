"""Large synchronous host calls are uploaded and detected in groups of frames: same results, counts and
readable levels as one call per frame, whatever the frames' layout in host memory."""
import numpy as np
import pytest

import oracle
from paper_2003_13493_gb300 import synth, vio

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [(640, 480), (752, 480), (1280, 720), (1021, 765)]


def layout(imgs, how):
    if how == "pageable":
        return imgs, None
    if how == "apart":  # every frame padded and far from the next: a copy each
        hold = [torch.empty((im.shape[0], im.shape[1] + 301), dtype=torch.uint8) for im in imgs]
        out = [h.numpy()[:, :im.shape[1]] for h, im in zip(hold, imgs)]
        for o, im in zip(out, imgs):
            o[...] = im
        return out, hold
    # one pinned ring, rows padded to 16 bytes; "mixed": every fifth frame unaligned, so spans end there
    room = [-(-im.shape[1] // 16) * 16 * im.shape[0] + 256 for im in imgs]
    ring = torch.zeros(sum(room), dtype=torch.uint8, pin_memory=True)
    out, at = [], 0
    for i, (im, r) in enumerate(zip(imgs, room)):
        pitch = -(-im.shape[1] // 16) * 16
        off = at + (3 if how == "mixed" and i % 5 == 4 else 0)
        v = ring.numpy()[off:off + pitch * im.shape[0]].reshape(im.shape[0], pitch)[:, :im.shape[1]]
        v[...] = im
        out.append(v)
        at += -(-r // 16) * 16 if i + 1 < len(imgs) else 0
    return out, ring


@pytest.mark.parametrize("how", ["ring", "mixed", "apart", "pageable"])
@pytest.mark.parametrize("levels", [1, 3])
@pytest.mark.parametrize("n", [2, 23])
def test_groups_match_single_frames(how, levels, n):
    sizes = [(3000, 1500)] * 2 if n == 2 else [SIZES[i % 4] for i in range(n)]
    imgs = [synth.make_frame(w, h, seed=i + 3) for i, (w, h) in enumerate(sizes)]
    frames, hold = layout(imgs, how)
    det = vio.Detector(max_frames=n)
    for _ in range(2):
        outs, counts = det.detect_host(frames, 15, 9, 32, levels)
    for i in sorted({0, 1, n // 2, n - 2, n - 1}):
        for k, want in enumerate(oracle.pyramid(imgs[i], levels)):
            assert np.array_equal(det.copy_level(i, k), want), (i, k)
    for i, im in enumerate(imgs):
        want, c = oracle.detect(im, 15, 9, 32, levels)
        assert np.array_equal(outs[i], want) and counts[i] == c, i
    det.close()


def test_a_budget_that_held_one_call_holds_the_groups():
    """Grouping takes no more device memory: the smallest budget that fits a profiled (ungrouped) call fits it."""
    imgs = [synth.make_frame(1280, 720, seed=i) for i in range(12)]
    frames, hold = layout(imgs, "ring")

    def works(budget, profile):
        try:
            det = vio.Detector(max_frames=12, mem_budget_bytes=budget, profile=profile)
            outs, _ = det.detect_host(frames, 15, 9, 32, 3)
            det.close()
            return outs
        except vio.VioError:
            return None

    lo, hi = 1 << 20, 64 << 20
    while hi - lo > 65536:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if works(mid, True) is not None else (mid, hi)
    a, b = works(hi, True), works(hi, False)
    assert b is not None and all(np.array_equal(x, y) for x, y in zip(a, b))


def test_a_call_that_fails_within_its_groups_leaves_the_context_usable():
    """The cell keys are a call's last buffer: just below the smallest budget a group fails after its copy began."""
    imgs = [synth.make_frame(1280, 720, seed=i) for i in range(12)]
    small = synth.make_frame(320, 240, seed=77)
    frames, hold = layout(imgs, "ring")

    def detector(budget):
        return vio.Detector(max_frames=12, mem_budget_bytes=budget)

    lo, hi = 1 << 20, 64 << 20
    while hi - lo > 1024:
        mid = (lo + hi) // 2
        try:
            det = detector(mid)
            det.detect_host(frames, 15, 9, 32, 3)
            det.close()
            hi = mid
        except vio.VioError:
            lo = mid
    det = detector(hi - 4096)
    with pytest.raises(vio.VioError):
        det.detect_host(frames, 15, 9, 32, 3)
    outs, counts = det.detect_host([small], 15, 9, 32, 3)
    want, c = oracle.detect(small, 15, 9, 32, 3)
    assert np.array_equal(outs[0], want) and counts[0] == c
    det.close()
