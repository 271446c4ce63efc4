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
    (400, 65532, 16, PIXEL, False), (400, 65532, 12, PIXEL, True), (600, 30000, 16, PIXEL, True),
])
def test_plans(h, w, nbins, layout, two):
    with ihist.Plan(h, w, nbins, layout) as plan:
        assert ihist.two_launch_plan(plan.handle) == two


@pytest.mark.parametrize("h,w,nbins,two", [(2160, 3840, 256, True), (3000, 4000, 128, True), (3000, 4000, 192, False)])
def test_table_plans(h, w, nbins, two):
    with ihist.Plan(h, w, nbins, bin_of_value=[v * nbins // 256 for v in range(256)]) as plan:
        assert ihist.two_launch_plan(plan.handle) == two
