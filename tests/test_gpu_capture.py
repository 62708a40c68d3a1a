"""Detections inside a caller's stream capture are refused, whichever kernels would take the call, and the context
stays usable.  (In a child process: the capture ends invalid.)"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import numpy as np, torch
import oracle
from paper_2003_13493_gb300 import synth, vio
pad = int(sys.argv[1])
img = synth.make_frame(752, 480, seed=5)
frame = torch.zeros((480, 752 + pad), dtype=torch.uint8, device="cuda")[:, :752]
frame.copy_(torch.from_numpy(img))
det, s = vio.Detector(max_frames=4), torch.cuda.Stream()
outs = [torch.empty((vio.num_cells(752, 480, 32), 4), dtype=torch.int32, device="cuda")]
counts = torch.empty(1, dtype=torch.int32, device="cuda")
torch.cuda.synchronize()
call = lambda: det.detect([frame], 20, 9, 32, 3, outs=outs, counts=counts, stream=s)
call(); call(); det.sync(s)
refused = False
try:
    with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s, capture_error_mode="thread_local"):
        try:
            call()
        except vio.VioError as e:
            refused = e.status == 3
except RuntimeError:
    pass
assert refused
outs[0].fill_(7)
torch.cuda.synchronize()
call()
det.sync(s)
want, n = oracle.detect(img, 20, 9, 32, 3)
assert np.array_equal(outs[0].cpu().numpy(), want) and int(counts[0]) == n
print("capture refused ok")
"""


@pytest.mark.parametrize("pad", [0, 1])
def test_a_capture_is_refused(pad):
    r = subprocess.run([sys.executable, "-c", CHILD, str(pad)], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "capture refused ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
