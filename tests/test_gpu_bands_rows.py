"""The two-launch path at the sizes where its band height follows from the
pixels: single frames on both sides of the line, batches across it, rebound
batches that keep their band height.  Equal to the look-back kernel word for
word (counts are integers: no tolerance)."""
import pytest

from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FUSED = {"ctas_per_sm": 32}  # the look-back kernel at its default tiling


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    ihist.load()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("h,w,nbins", [(169, 65000, 3), (170, 65033, 5), (1009, 11111, 4), (999, 11000, 12)])
@pytest.mark.parametrize("layout", [ihist.IHIST_BIN_MAJOR, ihist.IHIST_QUAD_MAJOR])
def test_frames_around_the_line(h, w, nbins, layout):
    nbins = (nbins + 3) // 4 * 4 if layout == ihist.IHIST_QUAD_MAJOR else nbins
    img = torch.from_numpy(synth.uniform_frame(h + w, h, w)).cuda()
    with ihist.Plan(h, w, nbins, layout) as plan, ihist.Plan(h, w, nbins, layout, tune=FUSED) as fused:
        assert ihist.two_launch_plan(plan.handle) and not ihist.two_launch_plan(fused.handle)
        assert torch.equal(plan.compute(img), fused.compute(img))
        assert plan.status() == ihist.IHIST_OK and fused.status() == ihist.IHIST_OK


@pytest.mark.parametrize("n", [34, 37])  # 10.4 and 11.4 million pixels
def test_batches_across_the_line(n):
    specs = [(480, 640, 2 + i % 3, 0) for i in range(n)]
    dev = [torch.from_numpy(synth.uniform_frame(i, 480, 640)).cuda() for i in range(n)]
    bins, layouts = [s[2] for s in specs], [0] * n
    with ihist.Batch(dev, bins, layouts) as batch, ihist.Batch(dev, bins, layouts, tune=FUSED) as fused:
        assert ihist.two_launch_batch(batch.handle) and not ihist.two_launch_batch(fused.handle)
        for frames in (dev, [f[:399, :517] for f in dev[:5]]):
            m = len(frames)
            for b in (batch, fused):
                outs = [torch.full((bins[i], *f.shape), -1, dtype=torch.int32, device="cuda")
                        for i, f in enumerate(frames)]
                b.set_io(frames, outs, bins[:m], layouts[:m])
                b.compute()
                assert b.status() == ihist.IHIST_OK
            assert all(torch.equal(x, y) for x, y in zip(batch.outs, fused.outs))
