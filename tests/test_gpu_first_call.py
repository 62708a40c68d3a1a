"""A context's first call and a call that needs more memory, on a stream that the default stream is not ordered with,
while the default stream is busy."""
import numpy as np
import pytest

import oracle
from paper_2003_13493_gb300 import synth, vio

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("pin", [False, True])
def test_first_call_beside_a_busy_default_stream(pin):
    imgs = [synth.make_frame(640, 480, seed=i) for i in range(12)]
    frames = [torch.from_numpy(im).cuda() for im in imgs]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)  # some 50 ms of work on the default stream
    det = vio.Detector(max_frames=16)
    if pin:
        det.set_variant(vio.variant_ids(1)[0])
    for n in (1, 12):  # the second call needs twelve times the keys
        with torch.cuda.stream(side):
            outs, counts = det.detect(frames[:n], 15, 9, 32, 3, stream=side)
        det.sync(side)
        torch.cuda._sleep(20_000_000)
        with torch.cuda.stream(side):
            got = [o.cpu().numpy() for o in outs]
            cnt = counts.cpu().numpy()
        for i in range(n):
            want, c = oracle.detect(imgs[i], 15, 9, 32, 3)
            assert np.array_equal(got[i], want) and cnt[i] == c, i
    det.close()
    torch.cuda.synchronize()
