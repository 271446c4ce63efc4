"""The checked build guards the two-launch path's workspace: CTAs with indices
outside the frame latch IHIST_ERR_CHECK_FAILED and access nothing, and the
frame's own CTAs leave the histogram exact.  The buffers are larger than the
frame needs, so that no access of either build lies outside an allocation."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1711_01919_gb300 import build as cuda_build
from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MARGIN = 1 << 20  # bytes on both sides of the workspace and of the output


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "band_guard_probe.cu")
    cmd = [cuda_build.nvcc(), *cuda_build.ARCH, *cuda_build.NVCC_FLAGS, "-DIHIST_CHECKED", "-I", cuda_build.CSRC,
           "-shared", src, "-o", lib]
    subprocess.run(cmd, check=True, capture_output=True, timeout=600)
    so = ctypes.CDLL(lib)
    so.probe_workspace.restype = ctypes.c_size_t
    vp, ci = ctypes.c_void_p, ctypes.c_int
    so.probe_run.argtypes = [ci] * 5 + [vp] * 4 + [ci] * 2
    return so


@pytest.mark.parametrize("layout", [ihist.IHIST_BIN_MAJOR, ihist.IHIST_QUAD_MAJOR, ihist.IHIST_PIXEL_MAJOR])
@pytest.mark.parametrize("h,w,nbins,R", [(70, 300, 12, 8), (200, 1300, 8, 32), (33, 131, 72, 16)])
def test_surplus_ctas_are_latched_and_touch_nothing(probe, h, w, nbins, R, layout):
    img = synth.uniform_frame(h + w, h, w)
    ref = oracle.integral_histogram(img, nbins)
    if layout == ihist.IHIST_QUAD_MAJOR:
        ref = ref.reshape(nbins // 4, 4, h, w).transpose(0, 2, 3, 1)
    elif layout == ihist.IHIST_PIXEL_MAJOR:
        ref = ref.transpose(1, 2, 0)
    frame = torch.from_numpy(img).cuda()
    ws_bytes, out_bytes = probe.probe_workspace(h, w, nbins, layout, R), h * w * nbins * 4
    for chunks, bands in ((0, 0), (1, 0), (0, 1), (2, 3)):
        ws = torch.full((MARGIN + ws_bytes + MARGIN,), 0xa5, dtype=torch.uint8, device="cuda")
        out = torch.full((MARGIN + out_bytes + MARGIN,), 0xa5, dtype=torch.uint8, device="cuda")
        ctrl = torch.zeros(64, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        status = probe.probe_run(h, w, nbins, layout, R, frame.data_ptr(), out.data_ptr() + MARGIN,
                                 ws.data_ptr() + MARGIN, ctrl.data_ptr(), chunks, bands)
        assert status == (ihist.IHIST_ERR_CHECK_FAILED if chunks or bands else ihist.IHIST_OK), (chunks, bands)
        for buf, n in ((ws, ws_bytes), (out, out_bytes)):
            assert int((buf[:MARGIN] != 0xa5).sum()) == 0 and int((buf[MARGIN + n:] != 0xa5).sum()) == 0
        got = out[MARGIN:MARGIN + out_bytes].cpu().numpy().view(np.uint32).reshape(ref.shape)
        assert np.array_equal(got, ref), (chunks, bands)
