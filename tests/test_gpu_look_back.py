"""The look-back kernel under the calls whose default is the two-launch path:
a tiling selects it, and so does capturing a batch.  Each test asserts which
path ran.  Both paths of a batch share its slots' memory, so live and replayed
launches also follow each other.  Counts are integers: no tolerance."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

TILED = {"ctas_per_sm": 32}  # the kernel's own default tiling


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    ihist.load()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def u32(t):
    return t.cpu().numpy().view(np.uint32)


def reference(img, nbins, layout, table=None, joint=None):
    if joint is not None:
        r = oracle.integral_histogram_joint(img, joint)
    elif table is not None:
        r = oracle.integral_histogram_mapped(img, np.asarray(table, np.int32), nbins)
    else:
        r = oracle.integral_histogram(img, nbins)
    if layout == ihist.IHIST_PIXEL_MAJOR:
        return np.ascontiguousarray(r.transpose(1, 2, 0))
    if layout == ihist.IHIST_QUAD_MAJOR:
        b, h, w = r.shape
        return np.ascontiguousarray(r.reshape(b // 4, 4, h, w).transpose(0, 2, 3, 1))
    return r


def check(batch, refs):
    assert batch.status() == ihist.IHIST_OK
    for i, ref in enumerate(refs):
        assert np.array_equal(u32(batch.outs[i]).reshape(ref.shape), ref), i


def mixed(kind, seed):
    """Frames, bin counts, layouts, tables, joint bins and results of a batch."""
    specs = {  # (h, w, bins, layout, table or None, joint bins or None)
        "uniform": [(37, 131, 16, 0, 0, None), (240, 320, 12, 1, 0, None), (90, 250, 12, 2, 0, None),
                    (100, 1000, 64, 0, 0, None), (5, 3, 3, 1, 0, None)],
        "table": [(270, 480, 5, 0, 1, None), (64, 257, 7, 1, 0, None), (100, 1000, 8, 1, 1, None),
                  (50, 300, 16, 2, 1, None)],
        "joint": [(150, 300, 64, 0, 0, [4, 4, 4]), (64, 257, 16, 1, 0, [8, 2]), (61, 129, 30, 0, 0, None),
                  (120, 250, 16, 2, 0, [4, 2, 2])],
    }[kind]
    imgs, tables, joint, refs = [], [], [], []
    for i, (h, w, b, l, t, j) in enumerate(specs):
        imgs.append(synth.uniform_frame(seed + i, h, w) if j is None else
                    np.random.default_rng(seed + i).integers(0, 256, size=(h, w, len(j)), dtype=np.uint8))
        tables.append([(v * 7 + seed) % (b + 1) - 1 for v in range(256)] if t else None)
        joint.append(j)
        refs.append(reference(imgs[-1], b, l, tables[-1], j))
    dev = [torch.from_numpy(x).cuda() for x in imgs]
    return dev, [s[2] for s in specs], [s[3] for s in specs], tables, joint, refs


def make(data, tune):
    dev, nbins, layouts, tables, joint, _ = data
    return ihist.Batch(dev, nbins, layouts, tune=tune, tables=tables if any(tables) else None,
                       joint=joint if any(joint) else None)


@pytest.mark.parametrize("kind", ["uniform", "table", "joint"])
@pytest.mark.parametrize("tune", [None, TILED, {"rows_per_band": 9}])
def test_batches_of_every_binning_on_either_path(kind, tune):
    data = mixed(kind, 300)
    with make(data, tune) as batch:
        assert ihist.two_launch_batch(batch.handle) == (tune is None)
        for _ in range(2):
            batch.compute()
        check(batch, data[5])


@pytest.mark.parametrize("kind", ["uniform", "table", "joint"])
def test_live_and_replayed_launches_of_one_batch(kind):
    a, b = mixed(kind, 400), mixed(kind, 500)
    with make(a, None) as batch:
        batch.compute()  # live: the two-launch path
        check(batch, a[5])
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=side):
            batch.compute()  # captured: the look-back kernel
        # (a captured joint batch bins the frames it was captured with, so it is not bound anew)
        for data in (a,) if kind == "joint" else (a, b, a):
            batch.set_io(data[0], batch.outs, data[1], data[2], tables=data[3], joint=data[4])
            torch.cuda.synchronize()
            for launch in (graph.replay, batch.compute, batch.compute, graph.replay, graph.replay):
                for o in batch.outs:
                    o.fill_(-1)
                launch()
                torch.cuda.synchronize()
                check(batch, data[5])


@pytest.mark.parametrize("tune", [None, TILED])
def test_unaligned_frames(tune):
    imgs = [synth.uniform_frame(7 + i, 90, 300) for i in range(3)]
    dev = []
    for img in imgs:
        v = torch.zeros(1 + 90 * 311 + 16, dtype=torch.uint8, device="cuda")[1:1 + 90 * 311].view(90, 311)[:, :300]
        v.copy_(torch.from_numpy(img))
        dev.append(v)
    with ihist.Batch(dev, [12, 5, 64], [0, 1, 0], tune=tune) as batch:
        assert ihist.two_launch_batch(batch.handle) == (tune is None)
        batch.compute()
        check(batch, [reference(x, b, l) for x, b, l in zip(imgs, [12, 5, 64], [0, 1, 0])])


@pytest.mark.parametrize("tune", [None, TILED])
def test_default_launch_behind_a_kernel_that_writes_the_frame(tune):
    h, w, nbins = 1080, 1920, 16
    base = synth.gradient_frame(800, h, w)
    rects = synth.rects(801, 500, h, w)
    d, d_r = torch.from_numpy(base).cuda(), torch.from_numpy(rects).cuda()
    d_r2 = torch.empty_like(d_r)
    with ihist.Plan(h, w, nbins, tune=tune) as plan:
        assert ihist.two_launch_plan(plan.handle) == (tune is None)
        out = plan.empty_output()
        for key in (0x5a, 0x33, 0xff):
            frame = torch.bitwise_xor(d, key)
            plan.compute(frame, out)
            d_r2.copy_(d_r.flip(0))
            rows = plan.query(out, d_r2)
            torch.cuda.synchronize()
            ref = oracle.integral_histogram(base ^ key, nbins)
            assert np.array_equal(u32(out).reshape(plan.out_shape), ref)
            assert np.array_equal(u32(rows), oracle.query(ref, np.ascontiguousarray(rects[::-1])))
        assert plan.status() == ihist.IHIST_OK


@pytest.mark.parametrize("tune", [None, TILED])
def test_binnings_of_single_frames_on_either_path(tune):
    img = synth.uniform_frame(5, 90, 500)
    rgb = np.random.default_rng(3).integers(0, 256, size=(60, 300, 3), dtype=np.uint8)
    for kw, x, ref in (({"edges": [0, 10, 11, 100, 255]}, img,
                        oracle.integral_histogram_edges(img, [0, 10, 11, 100, 255])),
                       ({"bins_per_channel": [4, 4, 4]}, rgb, oracle.integral_histogram_joint(rgb, [4, 4, 4]))):
        with ihist.Plan(x.shape[0], x.shape[1], tune=tune, **kw) as plan:
            assert ihist.two_launch_plan(plan.handle) == (tune is None)
            got = plan.compute(torch.from_numpy(x).cuda())
            assert plan.status() == ihist.IHIST_OK
            assert np.array_equal(u32(got).reshape(ref.shape), ref)


def test_these_calls_in_the_checked_build():
    """The binnings and batches above once more with every work item, carry
    index and store of the look-back kernel guarded."""
    from paper_1711_01919_gb300 import build as cuda_build
    lib = cuda_build.build(checked=True)
    env = dict(os.environ, IHIST_LIB=lib)
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider", os.path.abspath(__file__),
                        "-k", "either_path or unaligned or replayed"], env=env, cwd=ROOT, capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0 and " passed" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
