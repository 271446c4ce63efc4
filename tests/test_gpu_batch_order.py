"""Batches whose bindings and launches are on different streams.  A launch's
grid comes from the binding it was made for, its descriptors from device
memory, so it runs after its binding's copies and before the next binding's,
wherever these were queued."""
import numpy as np
import pytest

import oracle
from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

HOLD = 200_000_000  # clock cycles a side stream is kept busy, about 0.1 s


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    ihist.load()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def bound(specs, seed):
    imgs = [synth.uniform_frame(seed + i, h, w) for i, (h, w, b, l) in enumerate(specs)]
    dev = [torch.from_numpy(x).cuda() for x in imgs]
    outs = [torch.full(ihist.out_shape(*s), -1, dtype=torch.int32, device="cuda") for s in specs]
    return imgs, dev, outs


def exact(imgs, outs, specs):
    for img, out, (h, w, b, l) in zip(imgs, outs, specs):
        ref = oracle.integral_histogram(img, b)
        if l == ihist.IHIST_PIXEL_MAJOR:
            ref = ref.transpose(1, 2, 0)
        if not np.array_equal(out.cpu().numpy().view(np.uint32), ref):
            return False
    return True


LARGE = [(240, 320, 16, 0), (300, 200, 8, 1), (200, 333, 32, 0)]
SMALL = [(40, 200, 8, 0)]


@pytest.mark.parametrize("first,second", [(SMALL, LARGE), (LARGE, SMALL)])
def test_a_launch_waits_for_its_bindings_copies(first, second):
    imgs, dev, outs = bound(second, 10)
    old_imgs, old_dev, old_outs = bound(first, 20)
    _, slots, slot_outs = bound(LARGE, 30)
    side = torch.cuda.Stream()
    with ihist.Batch(slots, [s[2] for s in LARGE], [s[3] for s in LARGE], outs=slot_outs) as batch:
        batch.set_io(old_dev, old_outs, [s[2] for s in first], [s[3] for s in first])
        batch.compute()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(HOLD)  # the copies below are made after it
        batch.set_io(dev, outs, [s[2] for s in second], [s[3] for s in second], stream=side)
        assert not side.query()
        batch.compute()
        torch.cuda.current_stream().synchronize()
        assert batch.status() == ihist.IHIST_OK
        assert exact(imgs, outs, second) and exact(old_imgs, old_outs, first)


@pytest.mark.parametrize("first,second", [(SMALL, LARGE), (LARGE, SMALL)])
def test_the_next_bindings_copies_wait_for_a_launch(first, second):
    imgs, dev, outs = bound(second, 40)
    old_imgs, old_dev, old_outs = bound(first, 50)
    _, slots, slot_outs = bound(LARGE, 60)
    side, third = torch.cuda.Stream(), torch.cuda.Stream()
    with ihist.Batch(slots, [s[2] for s in LARGE], [s[3] for s in LARGE], outs=slot_outs) as batch:
        batch.set_io(old_dev, old_outs, [s[2] for s in first], [s[3] for s in first])
        torch.cuda.synchronize()
        torch.cuda._sleep(HOLD)
        batch.compute()  # has not run when the next binding is made
        batch.set_io(dev, outs, [s[2] for s in second], [s[3] for s in second], stream=side)
        assert not torch.cuda.current_stream().query()
        batch.compute(stream=third)
        batch.compute(stream=side)
        torch.cuda.synchronize()
        assert batch.status() == ihist.IHIST_OK
        assert exact(old_imgs, old_outs, first) and exact(imgs, outs, second)


def test_upload_compute_on_other_streams_follows_the_last_launch():
    specs = LARGE
    imgs, dev, outs = bound(specs, 70)
    new = [torch.from_numpy(synth.gradient_frame(80 + i, h, w)).pin_memory() for i, (h, w, b, l) in enumerate(specs)]
    side, copy = torch.cuda.Stream(), torch.cuda.Stream()
    with ihist.Batch(dev, [s[2] for s in specs], [s[3] for s in specs], outs=outs) as batch:
        torch.cuda._sleep(HOLD)
        batch.compute()  # reads the frames that the upload below replaces
        batch.set_io(dev, [torch.empty_like(o) for o in outs], [s[2] for s in specs], [s[3] for s in specs])
        batch.upload_compute(new, stream=side, copy_stream=copy)
        torch.cuda.synchronize()
        assert batch.status() == ihist.IHIST_OK
        assert exact(imgs, outs, specs)
        assert exact([x.numpy() for x in new], batch.outs, specs)


def test_a_captured_binding_leaves_live_launches_to_the_look_back_kernel():
    imgs, dev, outs = bound(LARGE, 90)
    s_imgs, s_dev, s_outs = bound(SMALL, 95)
    side = torch.cuda.Stream()
    with ihist.Batch(dev, [s[2] for s in LARGE], [s[3] for s in LARGE], outs=outs) as batch:
        batch.compute()
        torch.cuda.synchronize()
        assert ihist.two_launch_batch(batch.handle)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side, capture_error_mode="relaxed"):  # it waits for an event on the host
            batch.set_io(s_dev, s_outs, [s[2] for s in SMALL], [s[3] for s in SMALL])
        assert not ihist.two_launch_batch(batch.handle)
        graph.replay()
        batch.compute()
        assert batch.status() == ihist.IHIST_OK
        assert exact(imgs, outs, LARGE) and exact(s_imgs, s_outs, SMALL)
