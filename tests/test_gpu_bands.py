"""The two-launch path (count kernel, then emit kernel) that plans without a
tiling of their own take, in all three layouts: equal to the oracle,
and to the fused look-back kernel (a plan with a tiling), word for word, at
the edges of its tiles (rows per band 8, 16 and 32, superbands of 4 bands, 64
and 128 columns, segments of 8 chunks, 32 and 64 bins of a pixel's record), for every binning, pitched and
unaligned frames and unaligned outputs.  Counts are integers: no tolerance."""
import numpy as np
import pytest

import oracle
from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FUSED = {"ctas_per_sm": 32}  # the default tiling of the fused kernel


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    ihist.load()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def u32(t):
    return t.cpu().numpy().view(np.uint32)


def laid_out(ref, layout):
    if layout == ihist.IHIST_QUAD_MAJOR:
        b, h, w = ref.shape
        return np.ascontiguousarray(ref.reshape(b // 4, 4, h, w).transpose(0, 2, 3, 1))
    if layout == ihist.IHIST_PIXEL_MAJOR:
        return np.ascontiguousarray(ref.transpose(1, 2, 0))
    return ref


def on_gpu(img, pad=0, offset=0):
    """The frame on the device, rows pad bytes wider, starting offset bytes in."""
    h, row = img.shape[0], int(np.prod(img.shape[1:]))
    buf = torch.zeros(offset + h * (row + pad), dtype=torch.uint8, device="cuda")
    view = buf[offset:].view(h, row + pad)[:, :row]
    view.copy_(torch.from_numpy(img.reshape(h, row)))
    return view if img.ndim == 2 else view.unflatten(1, img.shape[1:])


def computed(plan, frame, shift=0):
    """H into a buffer that starts shift words past a 256-byte boundary, with
    canary words on both sides; twice, the second time over the first's counts."""
    n = plan.h * plan.w * plan.nbins
    buf = torch.full((64 + shift + n + 64,), -7, dtype=torch.int32, device="cuda")
    out = buf[64 + shift:64 + shift + n]
    plan.compute(frame, out)
    plan.compute(frame, out)
    assert plan.status() == ihist.IHIST_OK
    assert int((buf[:64 + shift] != -7).sum()) == 0 and int((buf[64 + shift + n:] != -7).sum()) == 0
    return u32(out).reshape(plan.out_shape)


@pytest.mark.parametrize("layout", [ihist.IHIST_BIN_MAJOR, ihist.IHIST_QUAD_MAJOR, ihist.IHIST_PIXEL_MAJOR])
@pytest.mark.parametrize("h,w,nbins", [
    (1, 1, 1), (7, 63, 4), (8, 64, 5), (9, 65, 12), (31, 127, 256), (32, 128, 253), (33, 129, 8), (65, 1023, 3),
    (64, 1024, 16), (127, 1025, 24), (129, 2049, 4), (257, 260, 64), (600, 640, 32), (2049, 130, 8), (2, 6000, 4),
    (140, 1921, 100), (40, 200, 72), (70, 161, 33)])
def test_edges_of_the_tiles(h, w, nbins, layout):
    if layout == ihist.IHIST_QUAD_MAJOR:
        nbins = (nbins + 3) // 4 * 4
    img = synth.uniform_frame(h * 7919 + w + nbins, h, w)
    ref = laid_out(oracle.integral_histogram(img, nbins), layout)
    for pad, offset, shift in ((0, 0, 0), (3, 1, 1), (16 - w % 16, 0, 4), (5, 2, 2)):
        with ihist.Plan(h, w, nbins, layout) as plan:
            got = computed(plan, on_gpu(img, pad, offset), shift)
        assert np.array_equal(got, ref), (pad, offset, shift)


@pytest.mark.parametrize("layout", [ihist.IHIST_BIN_MAJOR, ihist.IHIST_QUAD_MAJOR, ihist.IHIST_PIXEL_MAJOR])
@pytest.mark.parametrize("h,w", [(33, 200), (300, 1100)])
@pytest.mark.parametrize("nbins", [4, 252, 256])
def test_tables_with_values_in_no_bin(h, w, nbins, layout):
    img = synth.gradient_frame(h + w, h, w)
    table = [(v * 5) % (nbins + 1) - 1 for v in range(256)]
    ref = laid_out(oracle.integral_histogram_mapped(img, np.asarray(table, np.int32), nbins), layout)
    with ihist.Plan(h, w, nbins, layout, bin_of_value=table) as plan:
        assert np.array_equal(computed(plan, on_gpu(img, 5, 3), 3), ref)


@pytest.mark.parametrize("bins", [[256], [5, 7], [4, 4, 4], [2, 3, 2, 4]])
def test_joint_bins(bins):
    img = np.random.default_rng(len(bins)).integers(0, 256, size=(70, 261, len(bins)), dtype=np.uint8)
    ref = oracle.integral_histogram_joint(img, bins)
    for tune in (None, {"overlap": 1}):
        with ihist.Plan(70, 261, bins_per_channel=bins, tune=tune) as plan:
            assert np.array_equal(computed(plan, on_gpu(img, 7, 1)), ref)
            assert np.array_equal(computed(plan, on_gpu(img, -img[0].size % 4, 4)), ref)  # rows on 4-byte boundaries


@pytest.mark.parametrize("layout", [ihist.IHIST_BIN_MAJOR, ihist.IHIST_QUAD_MAJOR, ihist.IHIST_PIXEL_MAJOR])
@pytest.mark.parametrize("h,w,nbins", [(1080, 1920, 64), (1081, 1921, 20), (2100, 3000, 12), (240, 320, 16),
                                       (61, 40000, 8), (8192, 700, 8)])
@pytest.mark.parametrize("overlap", [0, 1])
def test_equals_the_fused_kernel(h, w, nbins, layout, overlap):
    """Several frames back to back through one plan, so that a frame's counts
    follow the previous frame's emit."""
    imgs = [on_gpu(synth.uniform_frame(h + w + i, h, w)) for i in range(3)]
    with ihist.Plan(h, w, nbins, layout, tune={"overlap": overlap}) as plan, \
            ihist.Plan(h, w, nbins, layout, tune=FUSED) as fused:
        outs = [plan.empty_output() for _ in imgs]
        torch.cuda.synchronize()
        for img, out in zip(imgs, outs):
            plan.compute(img, out)
        for img, out in zip(imgs, outs):
            assert torch.equal(out, fused.compute(img))
        assert plan.status() == ihist.IHIST_OK and fused.status() == ihist.IHIST_OK


def test_plans_of_different_bin_counts_side_by_side():
    """A plan made later, whose count kernel needs less shared memory, leaves
    an earlier plan's launches as they were."""
    img = synth.uniform_frame(11, 50, 300)
    with ihist.Plan(50, 300, 256) as wide, ihist.Plan(50, 300, 4) as narrow:
        for plan in (wide, narrow, wide):
            assert np.array_equal(computed(plan, on_gpu(img)), oracle.integral_histogram(img, plan.nbins))
