"""Batches of the two-launch path whose frames need count CTAs of different
shared memory: enough of them to be counted in a launch per size, and few
enough to share one.  Equal to the oracle, also after rebinding."""
import numpy as np
import pytest

import oracle
from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BINS = (8, 256, 72, 73, 100, 128, 180, 200, 16)  # all four numbers of CTAs per SM


@pytest.mark.parametrize("n", [9, 60, 300])
@pytest.mark.parametrize("tables", [False, True])
def test_mixed_bin_counts(n, tables):
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    specs = [(40 + i % 7, 130 + 8 * (i % 9), BINS[i % len(BINS)], (0, 1)[i % 2]) for i in range(n)]
    imgs = [synth.uniform_frame(i, h, w) for i, (h, w, b, l) in enumerate(specs)]
    tb = [[(v * 5) % (b + 1) - 1 for v in range(256)] if tables and b < 253 and i % 3 == 0 else None
          for i, (h, w, b, l) in enumerate(specs)]
    dev = [torch.from_numpy(x).cuda() for x in imgs]
    with ihist.Batch(dev, [s[2] for s in specs], [s[3] for s in specs], tables=tb if tables else None) as batch:
        assert ihist.two_launch_batch(batch.handle)
        outs = batch.outs
        for m in (n, n // 3, n):
            batch.set_io(dev[:m], outs[:m], [s[2] for s in specs[:m]], [s[3] for s in specs[:m]], tables=tb[:m])
            for o in batch.outs:
                o.fill_(-1)
            batch.compute()
            assert batch.status() == ihist.IHIST_OK
            for i in range(m):
                h, w, b, l = specs[i]
                ref = (oracle.integral_histogram(imgs[i], b) if tb[i] is None else
                       oracle.integral_histogram_mapped(imgs[i], np.asarray(tb[i], np.int32), b))
                ref = ref.transpose(1, 2, 0) if l else ref
                assert np.array_equal(batch.outs[i].cpu().numpy().view(np.uint32), ref), i
