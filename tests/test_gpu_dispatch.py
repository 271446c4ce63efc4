"""Which kernels an untuned plan or batch takes: shapes on both sides of each
line, each line where the two paths were measured to cross (ihist_bands.cu,
ihist_batch_api.cu)."""
import pytest

from paper_1711_01919_gb300 import ihist

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BIN, PIXEL, QUAD = ihist.IHIST_BIN_MAJOR, ihist.IHIST_PIXEL_MAJOR, ihist.IHIST_QUAD_MAJOR


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    ihist.load()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("h,w,nbins,layout,two", [
    # pixels and rows
    (480, 640, 32, BIN, True), (3000, 4000, 16, BIN, True), (3001, 4000, 16, BIN, False),
    (8192, 64, 8, BIN, True), (8193, 64, 8, BIN, False), (4320, 7680, 32, QUAD, True), (6400, 6400, 32, QUAD, False),
    # counts beyond L2, only where the look-back kernel's loads are whole
    (2160, 3840, 128, BIN, True), (2160, 3840, 192, BIN, False), (3000, 4000, 64, BIN, True),
    (3000, 4000, 128, BIN, False), (2999, 4001, 256, BIN, True), (8192, 1456, 128, BIN, True),
    (8192, 1456, 192, BIN, False), (8192, 1464, 256, BIN, True), (1080, 1920, 256, BIN, True),
    (4320, 7680, 64, QUAD, True), (4320, 7680, 128, QUAD, False), (4320, 5800, 256, QUAD, True),
    (4320, 7680, 256, PIXEL, True),
    # whole small records of large pixel-major frames
    (4320, 7680, 8, PIXEL, False), (4320, 7680, 6, PIXEL, True), (3000, 4000, 8, PIXEL, True),
    (600, 65532, 8, PIXEL, False), (600, 65535, 8, PIXEL, True), (8192, 4800, 4, QUAD, False), (4320, 7680, 4, QUAD, True),
    (400, 65532, 16, PIXEL, False), (400, 65532, 12, PIXEL, True), (600, 30000, 16, PIXEL, True),
])
def test_plans(h, w, nbins, layout, two):
    with ihist.Plan(h, w, nbins, layout) as plan:
        assert ihist.two_launch_plan(plan.handle) == two


@pytest.mark.parametrize("h,w,nbins,two", [(2160, 3840, 256, True), (3000, 4000, 128, True), (3000, 4000, 192, False)])
def test_table_plans(h, w, nbins, two):
    with ihist.Plan(h, w, nbins, bin_of_value=[v * nbins // 256 for v in range(256)]) as plan:
        assert ihist.two_launch_plan(plan.handle) == two


@pytest.mark.parametrize("n,h,w,nbins,layout,two", [
    # output bytes of aligned bin-major frames
    (32, 1080, 1920, 64, BIN, True), (33, 1080, 1920, 64, BIN, False), (33, 1080, 1920, 64, QUAD, True),
    # pixels of frames with few bins, by layout and width
    (16, 1080, 1920, 4, BIN, True), (24, 1080, 1920, 4, BIN, False), (24, 1080, 1921, 4, BIN, True),
    (24, 1080, 1928, 4, BIN, True), (24, 1080, 1920, 8, BIN, True), (40, 1080, 1920, 8, BIN, False),
    (64, 1080, 1920, 16, BIN, False), (64, 1080, 1920, 20, BIN, True), (8, 2160, 3840, 4, BIN, True),
    (12, 2160, 3840, 4, BIN, False), (40, 1080, 1920, 8, QUAD, True), (64, 1080, 1920, 8, QUAD, False),
    (9, 1080, 1920, 8, PIXEL, True), (12, 1080, 1920, 8, PIXEL, False), (16, 1080, 1920, 4, PIXEL, True),
    (24, 1080, 1920, 4, PIXEL, False), (64, 1080, 1920, 9, PIXEL, True), (128, 720, 1280, 8, PIXEL, True),
    (6, 1081, 1921, 4, PIXEL, True), (8, 1081, 1921, 4, PIXEL, False), (24, 1081, 1921, 8, PIXEL, True),
])
def test_batches(n, h, w, nbins, layout, two):
    frame = torch.zeros((h, w), dtype=torch.uint8, device="cuda")
    out = torch.empty(ihist.out_shape(h, w, nbins, layout), dtype=torch.int32, device="cuda")
    with ihist.Batch([frame] * n, nbins, [layout] * n, outs=[out] * n) as batch:
        assert ihist.two_launch_batch(batch.handle) == two


def test_a_frame_of_another_kind_keeps_the_batch_in_two_launches():
    frame = torch.zeros((1080, 1920), dtype=torch.uint8, device="cuda")
    out = torch.empty(1080 * 1920 * 32, dtype=torch.int32, device="cuda")
    for extra in ((PIXEL, 32), (BIN, 256)):
        frames = [frame] * 40
        bins, layouts = [8] * 39 + [extra[1]], [BIN] * 39 + [extra[0]]
        outs = [out[:1080 * 1920 * 8].view(8, 1080, 1920)] * 39 + [
            torch.empty(ihist.out_shape(1080, 1920, extra[1], extra[0]), dtype=torch.int32, device="cuda")]
        with ihist.Batch(frames, bins, layouts, outs=outs) as batch:
            assert ihist.two_launch_batch(batch.handle)
