"""The persistent kernels where the tile kernel takes a context's ordinary calls: without graphs, with the device-side
index checks, and in groups of a host call.  (A pinned variant, or more than 64 frames, keeps a call with them.)"""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2003_13493_gb300 import synth, vio

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def check(det, imgs, frames, t, a, c, levels, score=0, radius=1):
    for _ in range(2):
        outs, counts = det.detect(frames, t, a, c, levels)
    det.sync()
    for i, im in enumerate(imgs):
        want, n = oracle.detect(im, t, a, c, levels, score, nms_radius=radius)
        assert np.array_equal(outs[i].cpu().numpy(), want) and int(counts[i]) == n, (im.shape, levels)


@pytest.mark.parametrize("score,radius", [(0, 1), (1, 1), (2, 1), (0, 2), (1, 3), (2, 4)])
def test_without_graphs(score, radius):
    imgs = [synth.make_frame(w, h, seed=w + i) for i, (w, h) in enumerate([(640, 480), (753, 481), (368, 187)])]
    pitched = [torch.zeros((im.shape[0], -(-im.shape[1] // 16) * 16), dtype=torch.uint8, device="cuda") for im in imgs]
    aligned = [p[:, :im.shape[1]] for p, im in zip(pitched, imgs)]
    for f, im in zip(aligned, imgs):
        f.copy_(torch.from_numpy(im))
    tight = [torch.from_numpy(im).cuda() for im in imgs]  # 753 columns: staged by the pyramid kernel
    det = vio.Detector(max_frames=8, use_graphs=False, score=score, nms_radius=radius)
    for v in vio.variant_ids(radius):
        det.set_variant(v)
        for levels in (1, 3, 5 if radius == 1 else 4):
            for frames in (aligned, tight):
                check(det, imgs, frames, 12, 9, 32, levels, score, radius)
    det.close()


CHILD = r"""
import numpy as np, torch, oracle
from paper_2003_13493_gb300 import synth, vio
assert vio.lib_path().endswith("libvio_gb300_checked.so")
imgs = synth.mixed_batch(first_seed=2, per_size=16)[::9] + [synth.make_frame(257, 131, seed=4)]
frames = [torch.from_numpy(i).cuda() for i in imgs]
for score, radius in [(1, 1), (2, 1), (0, 2), (1, 3), (0, 4), (2, 4)]:
    det = vio.Detector(max_frames=64, score=score, nms_radius=radius)
    for v in vio.variant_ids(radius):
        det.set_variant(v)
        for t, a in ((5, 9), (15, 12)):
            outs, counts = det.detect(frames, t, a, 32, 3)
            det.sync()  # raises when an index check fired
            for i, im in enumerate(imgs):
                want, n = oracle.detect(im, t, a, 32, 3, score, nms_radius=radius)
                assert np.array_equal(outs[i].cpu().numpy(), want) and int(counts[i]) == n, (score, radius, i)
    det.close()
print("checked build ok")
"""


def test_scores_and_radii_with_index_checks():
    from paper_2003_13493_gb300 import build

    build.build(checked=True)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, VIO_CHECKED="1", PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "checked build ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]


@pytest.mark.parametrize("levels", [1, 3])
@pytest.mark.parametrize("pinned_out", [False, True])
def test_groups_of_many_small_frames(levels, pinned_out):
    """260 frames of 160x120 are groups of 109, 109 and 42 frames: the persistent kernels twice, then the tile kernel,
    on the same keys and pyramid."""
    n, (w, h) = 260, (160, 120)
    imgs = [synth.make_frame(w, h, seed=i, n_shapes=6) for i in range(n)]
    ring = torch.empty((n, h, w), dtype=torch.uint8, pin_memory=True)
    for i, im in enumerate(imgs):
        ring[i].copy_(torch.from_numpy(im))
    cells = vio.num_cells(w, h, 32)
    outs = torch.empty((n, cells, 4), dtype=torch.int32, pin_memory=pinned_out)
    counts = torch.empty(n, dtype=torch.int32, pin_memory=pinned_out)
    batch = vio.HostBatch([ring[i].numpy() for i in range(n)], [outs[i].numpy() for i in range(n)], counts.numpy())
    det = vio.Detector(max_frames=n)
    for _ in range(2):
        outs.fill_(7)
        det.detect_host_batch(batch, 12, 9, 32, levels)
        for i, im in enumerate(imgs):
            want, c = oracle.detect(im, 12, 9, 32, levels)
            assert np.array_equal(outs[i].numpy(), want) and int(counts[i]) == c, i
    det._last_dims = [(w, h)] * n
    for i in (0, 1, 108, 109, 217, 218, 259):
        for k, want in enumerate(oracle.pyramid(imgs[i], levels)):
            assert np.array_equal(det.copy_level(i, k), want), (i, k)
    det.close()
