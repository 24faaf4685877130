"""Voxel silhouettes on the GPU (psfs_reproject) against the oracle's brute
force.  The GPU tests pixel-centre rays in float32, so a pixel whose ray
passes within ~1e-3 voxel of a cube edge may go either way: every pixel the
oracle sets with the cubes shrunk by GROW voxel sizes must be set, and every
pixel it leaves unset with the cubes grown by GROW must be unset."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1311_6811_gb300 import psfs  # noqa: E402
from synth import scene as S  # noqa: E402
from tests.gpu_helpers import to_dev  # noqa: E402

pytestmark = pytest.mark.gpu
GROW = 2e-3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    psfs.load()


def _gpu_masks(rec, lists, counts, stride):
    F = counts.numel()
    H, W = rec.image_shape[1], rec.image_shape[2]
    masks = torch.full((F, rec.n_cams, H, W), 7, dtype=torch.uint8, device="cuda")
    psfs.psfs_reproject(rec.handle, F, lists, stride, counts, masks)
    assert rec.sync() == psfs.PSFS_OK
    return masks.cpu().numpy()


def _check(grid, cams, lst, got):
    assert set(np.unique(got)) <= {0, 1}
    inner = oracle.reproject(grid, cams, lst, grow=-GROW)
    outer = oracle.reproject(grid, cams, lst, grow=GROW)
    assert np.all(got >= inner), int((got < inner).sum())
    assert np.all(got <= outer), int((got > outer).sum())
    return int((outer != inner).sum())


def test_random_sets_and_a_box():
    sc = S.make_scene(seed=41, grid_n=24, cube_side=2.0, n_cams=3, width=64, height=48, focal=60.0)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    V = sc.grid.n_voxels
    rng = np.random.default_rng(1)
    box = np.zeros((24, 24, 24), bool)
    box[4:15, 6:20, 2:12] = True
    sets = [rng.choice(V, 40, replace=False), rng.choice(V, 400, replace=False), np.flatnonzero(box.ravel()),
            np.array([], np.int64)]
    stride = max(s.size for s in sets)
    lists = torch.zeros((len(sets), stride), dtype=torch.int32)
    counts = torch.zeros((len(sets),), dtype=torch.int32)
    for f, s_ in enumerate(sets):
        lists[f, :s_.size] = torch.from_numpy(s_.astype(np.int32))
        counts[f] = s_.size
    got = _gpu_masks(rec, lists.cuda(), counts.cuda(), stride)
    for f, s_ in enumerate(sets):
        _check(sc.grid, sc.cams, s_.astype(np.uint32), got[f])
    assert got[2].sum() > 500 and got[3].sum() == 0
    rec.close()


def test_reconstructed_surface_silhouettes():
    """A walking sequence: the silhouettes of each frame's surface list (and,
    for one frame, of its full occupied list) against the oracle."""
    sc = S.make_scene(seed=42, grid_n=32, cube_side=2.0, n_cams=4, width=96, height=72, focal=90.0,
                      n_frames=3, walking=True)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    rec.set_background(to_dev(sc.mean), to_dev(sc.var))
    imgs = to_dev(sc.images)
    F, V = imgs.shape[0], rec.n_voxels
    occ = torch.empty((F, V), device="cuda")
    lists = torch.empty((F, V), dtype=torch.int32, device="cuda")
    counts = torch.zeros((F,), dtype=torch.int32, device="cuda")
    psfs.psfs_reconstruct_sequence(rec.handle, F, imgs, occ, lists, V, counts)
    sl = torch.empty((F, V), dtype=torch.int32, device="cuda")
    sc_n = torch.zeros((F,), dtype=torch.int32, device="cuda")
    psfs.psfs_surface(rec.handle, F, lists, V, counts, sl, V, sc_n)
    got_s = _gpu_masks(rec, sl, sc_n, V)
    got_o = _gpu_masks(rec, lists, counts, V)
    for f in range(F):
        surf = sl[f, :int(sc_n[f])].cpu().numpy().astype(np.uint32)
        assert surf.size > 50
        _check(sc.grid, sc.cams, surf, got_s[f])
        # the solid and its surface: the same silhouette up to grazing rays
        assert (got_s[f] != got_o[f]).sum() <= 0.001 * got_o[f].size
    full0 = lists[0, :int(counts[0])].cpu().numpy().astype(np.uint32)
    _check(sc.grid, sc.cams, full0, got_o[0])
    rec.close()


def test_camera_inside_the_grid():
    """Cameras inside an 8 m grid: cubes next to or behind a camera take the
    whole-image path; the exact test still decides."""
    sc = S.make_scene(seed=14, grid_n=12, cube_side=8.0, n_cams=2, width=48, height=40, focal=40.0)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    V = sc.grid.n_voxels
    rng = np.random.default_rng(3)
    s_ = rng.choice(V, 200, replace=False).astype(np.int32)
    lists = torch.from_numpy(s_).cuda().view(1, -1)
    counts = torch.tensor([s_.size], dtype=torch.int32, device="cuda")
    got = _gpu_masks(rec, lists, counts, s_.size)
    _check(sc.grid, sc.cams, s_.astype(np.uint32), got[0])
    rec.close()


@pytest.mark.parametrize("width,height,n_set", [(66, 50, 300), (320, 240, 300)])
def test_staged_and_direct_paths(width, height, n_set):
    """A CTA stages its chunk of 256 voxels in shared memory when the union of
    their boxes fits 32 KB of 4-byte-aligned rows, and stores directly
    otherwise: rows not a multiple of 4 bytes wide (66 px, direct), scattered
    voxels in a 320 x 240 image (unions larger than 32 KB, direct) and a
    solid box in the same rig (staged chunks)."""
    sc = S.make_scene(seed=43, grid_n=24, cube_side=2.0, n_cams=3, width=width, height=height,
                      focal=0.9 * width)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    V = sc.grid.n_voxels
    rng = np.random.default_rng(4)
    box = np.zeros((24, 24, 24), bool)
    box[6:18, 8:16, 4:20] = True
    sets = [rng.choice(V, n_set, replace=False), np.flatnonzero(box.ravel())]
    stride = max(s.size for s in sets)
    lists = torch.zeros((len(sets), stride), dtype=torch.int32)
    counts = torch.zeros((len(sets),), dtype=torch.int32)
    for f, s_ in enumerate(sets):
        lists[f, :s_.size] = torch.from_numpy(s_.astype(np.int32))
        counts[f] = s_.size
    got = _gpu_masks(rec, lists.cuda(), counts.cuda(), stride)
    for f, s_ in enumerate(sets):
        _check(sc.grid, sc.cams, s_.astype(np.uint32), got[f])
        assert got[f].sum() > 100
    rec.close()


@pytest.mark.parametrize("width,height,n_cams,frames", [(67, 51, 2, 1), (33, 1, 1, 3), (1100, 760, 1, 1),
                                                        (67, 51, 3, 250)])
def test_bitmask_bands_and_clusters(width, height, n_cams, frames):
    """Masks whose bytes do not start 16-byte aligned (odd sizes), an image of
    more pixels than one CTA's bitmask holds (two bands), one mask shared by a
    cluster (few frames) and one CTA per mask (many frames)."""
    sc = S.make_scene(seed=44, grid_n=20, cube_side=2.0, n_cams=n_cams, width=width, height=height,
                      focal=0.9 * width)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    s_ = np.random.default_rng(5).choice(sc.grid.n_voxels, 60, replace=False).astype(np.int32)
    lists = torch.from_numpy(s_).cuda().repeat(frames, 1)
    counts = torch.full((frames,), s_.size, dtype=torch.int32, device="cuda")
    got = _gpu_masks(rec, lists, counts, s_.size)
    _check(sc.grid, sc.cams, s_.astype(np.uint32), got[0])
    assert (got == got[0]).all()
    rec.close()


@pytest.mark.parametrize("width,height,n_cams,frames,offset", [(67, 51, 2, 1, 0), (67, 51, 2, 3, 1), (33, 1, 1, 3, 3),
                                                               (64, 48, 3, 2, 2), (1100, 760, 1, 1, 0),
                                                               (1400, 1290, 1, 1, 1)])
def test_parts_of_the_list(width, height, n_cams, frames, offset):
    """Few masks and lists of more than 4096 entries: parts of the list, a CTA
    each, OR-ed into a zeroed mask (masks at any byte, rows of any length, two
    bands; frames with a short and an empty list in the same call).  The masks
    are the OR of those of the list's pieces, which a cluster per mask takes,
    against the oracle, and the bytes beside them stay; a captured call gives
    the same."""
    sc = S.make_scene(seed=45, grid_n=20, cube_side=2.0, n_cams=n_cams, width=width, height=height,
                      focal=0.9 * width)
    stream = torch.cuda.Stream()
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params, stream=stream)
    rng = np.random.default_rng(6)
    sizes = [5000, 300, 0][:frames]
    stride = 5001
    lists = torch.zeros((frames, stride), dtype=torch.int32)
    for f, n in enumerate(sizes):
        lists[f, :n] = torch.from_numpy(np.sort(rng.choice(sc.grid.n_voxels, n, replace=False)).astype(np.int32))
    n_bytes = frames * n_cams * height * width

    def run(l, s_, c, buf):
        psfs.psfs_reproject(rec.handle, frames, l, s_, c, buf[offset:offset + n_bytes])

    def masks(buf):
        assert (buf[:offset] == 7).all() and (buf[offset + n_bytes:] == 7).all()
        return buf[offset:offset + n_bytes].cpu().numpy().reshape(frames, n_cams, height, width)

    want = np.zeros((frames, n_cams, height, width), np.uint8)
    for a in range(0, max(sizes), 2500):
        counts = torch.tensor([min(max(n - a, 0), 2500) for n in sizes], dtype=torch.int32).cuda()
        buf = torch.full((offset + n_bytes + 5,), 7, dtype=torch.uint8, device="cuda")
        piece = lists[:, a:a + 2500].contiguous().cuda()
        torch.cuda.synchronize()
        run(piece, 2500, counts, buf)
        assert rec.sync() == psfs.PSFS_OK
        want |= masks(buf)
    counts = torch.tensor(sizes, dtype=torch.int32).cuda()
    dev = lists.cuda()
    bufs = [torch.full((offset + n_bytes + 5,), 7, dtype=torch.uint8, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    run(dev, stride, counts, bufs[0])
    assert rec.sync() == psfs.PSFS_OK
    got = masks(bufs[0])
    assert np.array_equal(got, want)
    if width < 1000:   # the brute force over the large image takes half a minute
        _check(sc.grid, sc.cams, lists[0, :sizes[0]].numpy().astype(np.uint32), got[0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        run(dev, stride, counts, bufs[1])
    with torch.cuda.stream(stream):
        graph.replay()
        graph.replay()
    assert rec.sync() == psfs.PSFS_OK
    assert np.array_equal(masks(bufs[1]), want)
    rec.close()


def _depths(grid, cam):
    """Least and largest depth of every voxel's eight corners in one camera."""
    z, y, x = np.meshgrid(np.arange(grid.nz), np.arange(grid.ny), np.arange(grid.nx), indexing="ij")
    i = np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.float64)
    corner = np.array([[a, b, c] for a in (0, 1) for b in (0, 1) for c in (0, 1)])
    X = np.asarray(grid.origin) + (i[:, None, :] + corner[None]) * grid.voxel_size
    d = X @ cam.R[2] + cam.t[2]
    return d.min(1), d.max(1)


@pytest.mark.parametrize("width,height,frames", [(48, 40, 1), (48, 40, 320), (1100, 760, 1),
                                                 (1400, 1290, 1)])
def test_cubes_at_and_behind_a_camera(width, height, frames):
    """Cameras inside an 8 m grid: cubes wholly behind one, cubes at its plane
    (several of one thread, and in rounds of the list beyond its 32nd), in one
    band and in two, against the oracle."""
    sc = S.make_scene(seed=46, grid_n=36, cube_side=8.0, n_cams=1, width=width, height=height, focal=0.8 * width)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    lo, hi = _depths(sc.grid, sc.cams[0])
    at, behind, front = (np.flatnonzero(m) for m in ((lo < 0) & (hi > 0), hi < 0, lo > 0))
    assert at.size > 800 and behind.size > 1000
    rng = np.random.default_rng(7)
    n = 800 if width < 1000 else 60
    s_ = np.concatenate([rng.choice(at, n, replace=False), rng.choice(behind, 100), rng.choice(front, 20)])
    s_ = rng.permutation(s_).astype(np.int32)
    if frames > 1:
        s_ = np.tile(s_, 40)   # more rounds of the list than a thread remembers
    lists = torch.from_numpy(s_).cuda().repeat(frames, 1)
    counts = torch.full((frames,), s_.size, dtype=torch.int32, device="cuda")
    got = _gpu_masks(rec, lists, counts, s_.size)
    _check(sc.grid, sc.cams, np.unique(s_).astype(np.uint32), got[0])
    assert (got == got[0]).all()
    rec.close()


def test_cubes_behind_a_camera_cost_no_more_than_those_in_front():
    """A cube behind a camera meets no ray: it must not be tested against every
    pixel (that took milliseconds; these lists take about 10 us each, and the
    bound of ten times leaves room for a disturbed run)."""
    sc = S.make_scene(seed=47, grid_n=64, cube_side=8.0, n_cams=1, width=320, height=240, focal=250.0)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    lo, hi = _depths(sc.grid, sc.cams[0])
    times = []
    for m in (lo > 1.0, hi < 0):
        s_ = np.flatnonzero(m)[:4000].astype(np.int32)
        lists, counts = torch.from_numpy(s_).cuda().view(1, -1), torch.tensor([s_.size], dtype=torch.int32).cuda()
        masks = torch.empty((1, 1, 240, 320), dtype=torch.uint8, device="cuda")
        best = 1e9
        for _ in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            psfs.psfs_reproject(rec.handle, 1, lists, s_.size, counts, masks)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert rec.sync() == psfs.PSFS_OK
    assert times[1] <= 10 * times[0], times
    rec.close()


def test_two_bands():
    """An image of more pixels than one CTA's bitmask holds (1.77 million): two
    bands of one mask, with one cluster per band (few frames) and one CTA (many),
    against the oracle."""
    width, height = 1400, 1290
    sc = S.make_scene(seed=44, grid_n=20, cube_side=2.0, n_cams=1, width=width, height=height, focal=0.9 * width)
    rec = psfs.Reconstructor(sc.grid, sc.cams, sc.params)
    s_ = np.random.default_rng(5).choice(sc.grid.n_voxels, 60, replace=False).astype(np.int32)
    for frames in (1, 160):
        lists = torch.from_numpy(s_).cuda().repeat(frames, 1)
        counts = torch.full((frames,), s_.size, dtype=torch.int32, device="cuda")
        got = _gpu_masks(rec, lists, counts, s_.size)
        _check(sc.grid, sc.cams, s_.astype(np.uint32), got[0])
        assert (got == got[0]).all()
    rec.close()
