"""Plans and batches made while the device has room for the look-back kernel's
carries but not for the two-launch path's counts: they are made all the same,
and take the look-back kernel."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TILED = {"ctas_per_sm": 32}
PIECE = 2 << 20  # device memory is handed out in pieces of this size


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    ihist.load()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


class Full:
    """All of the device allocated but `hole` bytes in one piece, past torch's
    allocator (whose cached blocks would blur the line)."""

    def __init__(self, hole):
        self.driver, self.held = ctypes.CDLL("libcuda.so.1"), []
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = self.take(hole)
        assert free
        for piece in (8 << 30, 512 << 20, 64 << 20, PIECE):
            while True:
                p = self.take(piece)
                if not p:
                    break
                self.held.append(p)
        self.driver.cuMemFree_v2(ctypes.c_uint64(free))

    def take(self, n):
        p = ctypes.c_uint64()
        return p.value if self.driver.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(n)) == 0 else 0

    def close(self):
        for p in self.held:
            self.driver.cuMemFree_v2(ctypes.c_uint64(p))


@pytest.mark.parametrize("kind", ["plan", "batch"])
def test_made_with_the_look_back_kernels_workspace(kind):
    h, w, nbins, n = 4320, 7680, 4, 16
    layout = ihist.IHIST_QUAD_MAJOR
    img = synth.uniform_frame(1, h, w) if kind == "plan" else synth.uniform_frame(2, 1080, 1920)
    frame = torch.from_numpy(img).cuda()
    out = torch.empty(img.size * 4, dtype=torch.int32, device="cuda")

    def make(tune=None):
        if kind == "plan":
            return ihist.Plan(h, w, nbins, layout, tune=tune)
        return ihist.Batch([frame] * n, nbins, [layout] * n, outs=[out.view(1, 1080, 1920, 4)] * n,
                           tune=tune)

    def nbytes(x):
        return x.workspace_bytes() if kind == "plan" else ihist.ihist_batch_workspace_bytes(x.handle)

    two = ihist.two_launch_plan if kind == "plan" else ihist.two_launch_batch
    with make() as a, make(TILED) as b:
        assert two(a.handle) and not two(b.handle)
        counts, carries = nbytes(a), nbytes(b)
    hole = carries + PIECE
    assert counts > hole + 2 * PIECE
    full = Full(hole)
    try:
        x = make()
        assert nbytes(x) < counts and not two(x.handle)
    finally:
        full.close()
    with x:
        got = (x.compute(frame, out) if kind == "plan" else x.compute()[0]).cpu().numpy().view(np.uint32)
        assert x.status() == ihist.IHIST_OK
        ref = oracle.integral_histogram(img, nbins)
        assert np.array_equal(got.reshape(*img.shape, 4), ref.transpose(1, 2, 0))
