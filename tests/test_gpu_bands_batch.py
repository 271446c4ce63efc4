"""Batches planned without a tiling go through the two-launch path (count
kernels, then emit kernels) where every frame fits it: results equal the
oracle word for word for mixed layouts, binnings, widths and alignments, for
more frames than one launch takes, across rebindings (also to frames that the
path does not take, which go back to the look-back kernel) and under graph
capture.  Counts are integers: no tolerance."""
import numpy as np
import pytest

import oracle
from paper_1711_01919_gb300 import ihist, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1711_01919_gb300 import build as cuda_build
    cuda_build.build()
    ihist.load()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


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


def check(batch, imgs, specs, tables=None, joint=None):
    assert batch.status() == ihist.IHIST_OK
    for i, (img, (h, w, b, l)) in enumerate(zip(imgs, specs)):
        ref = reference(img, b, l, tables and tables[i], joint and joint[i])
        got = batch.outs[i].cpu().numpy().view(np.uint32).reshape(ref.shape)
        assert np.array_equal(got, ref), (i, h, w, b, l)


def frames_of(specs, seed, joint=None):
    imgs = []
    for i, (h, w, b, l) in enumerate(specs):
        c = joint[i] if joint else None
        imgs.append(synth.uniform_frame(seed + i, h, w) if c is None else
                    np.random.default_rng(seed + i).integers(0, 256, size=(h, w, len(c)), dtype=np.uint8))
    return imgs, [torch.from_numpy(x).cuda() for x in imgs]


MIXED = [(1, 1, 3, 0), (37, 131, 16, 0), (33, 257, 40, 1), (64, 1024, 8, 2), (65, 1025, 5, 0), (100, 1300, 12, 1),
         (40, 2100, 64, 1), (31, 2050, 20, 2), (200, 90, 33, 0), (8, 128, 256, 1), (300, 320, 16, 0)]


@pytest.mark.parametrize("seed", [1, 2])
def test_mixed_layouts_and_rebinding(seed):
    imgs, dev = frames_of(MIXED, 100 * seed)
    with ihist.Batch(dev, [s[2] for s in MIXED], [s[3] for s in MIXED]) as batch:
        for _ in range(2):
            batch.compute()
        check(batch, imgs, MIXED)
        # smaller frames in other layouts, then the planned ones again
        small = [(max(1, h - 1), max(1, w - 3), b // 4 * 4 or 4, (l + 1) % 3) if b >= 4 else (1, 1, 1, 0)
                 for (h, w, b, l) in MIXED]
        s_imgs, s_dev = frames_of(small, 100 * seed + 50)
        outs = [torch.empty(ihist.out_shape(*s), dtype=torch.int32, device="cuda") for s in small]
        old = batch.outs
        batch.set_io(s_dev, outs, [s[2] for s in small], [s[3] for s in small])
        batch.compute()
        check(batch, s_imgs, small)
        batch.set_io(dev, old, [s[2] for s in MIXED], [s[3] for s in MIXED])
        batch.compute()
        check(batch, imgs, MIXED)


def test_tables_joint_and_uniform_frames():
    specs = [(50, 300, 5, 0), (64, 257, 256, 0), (70, 140, 252, 1), (33, 200, 8, 2)]
    tables = [ihist.edges_table([0, 16, 64, 128, 129, 256]), None, [(v * 5) % 253 - 1 for v in range(256)], None]
    imgs, dev = frames_of(specs, 7)
    with ihist.Batch(dev, [s[2] for s in specs], [s[3] for s in specs], tables=tables) as batch:
        batch.compute()
        check(batch, imgs, specs, tables=tables)
    specs = [(60, 300, 64, 0), (41, 129, 24, 1), (50, 100, 30, 0)]
    joint = [[4, 4, 4], [2, 4, 3], None]
    imgs, dev = frames_of(specs, 9, joint)
    with ihist.Batch(dev, [s[2] for s in specs], [s[3] for s in specs], joint=joint) as batch:
        batch.compute()
        check(batch, imgs, specs, joint=joint)


def test_table_of_256_bins_with_values_in_no_bin_takes_the_look_back_kernel():
    specs = [(40, 150, 256, 0), (30, 200, 16, 0)]
    tables = [[v if v % 7 else -1 for v in range(256)], None]
    imgs, dev = frames_of(specs, 21)
    with ihist.Batch(dev, [s[2] for s in specs], [s[3] for s in specs], tables=tables) as batch:
        batch.compute()
        check(batch, imgs, specs, tables=tables)


def test_more_frames_than_one_launch_takes():
    specs = [(8 + i % 5, 20 + i % 37, 1 + i % 9, (0, 1)[i % 2]) for i in range(300)]
    imgs, dev = frames_of(specs, 1000)
    with ihist.Batch(dev, [s[2] for s in specs], [s[3] for s in specs]) as batch:
        batch.compute()
        check(batch, imgs, specs)


def test_rebinding_to_a_frame_the_path_does_not_take():
    """A frame taller than the path's limit fits the slot's carries: the whole
    binding goes through the look-back kernel, and back again."""
    specs = [(2000, 600, 16, 0), (200, 300, 8, 0)]
    tall = [(9000, 100, 16, 0), (200, 300, 8, 0)]
    imgs, dev = frames_of(specs, 31)
    t_imgs, t_dev = frames_of(tall, 41)
    with ihist.Batch(dev, [16, 8]) as batch:
        batch.compute()
        check(batch, imgs, specs)
        old = batch.outs
        outs = [torch.empty(ihist.out_shape(*s), dtype=torch.int32, device="cuda") for s in tall]
        batch.set_io(t_dev, outs, [16, 8], [0, 0])
        batch.compute()
        check(batch, t_imgs, tall)
        batch.set_io(dev, old, [16, 8], [0, 0])
        batch.compute()
        check(batch, imgs, specs)


def test_captured_launches_follow_later_bindings():
    specs = [(120, 256, 8, 0), (60, 128, 16, 0)]
    imgs, dev = frames_of(specs, 51)
    with ihist.Batch(dev, [8, 16]) as batch:
        batch.compute()
        check(batch, imgs, specs)
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=side):
            batch.compute()
        small = [(100, 256, 8, 0), (60, 128, 12, 0)]
        s_imgs, s_dev = frames_of(small, 61)
        outs = [torch.empty(ihist.out_shape(*s), dtype=torch.int32, device="cuda") for s in small]
        batch.set_io(s_dev, outs, [8, 12], [0, 0])
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        check(batch, s_imgs, small)
