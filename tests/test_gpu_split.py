"""GPU checks of deferred shading through the task workspace (the split march): images and
sample counts equal the per-ray schedule's bit for bit, when the workspace is small and goes
through several rounds, gives tiles up and takes them up again, in bands of rows, and leaves
dense tiles to the single-kernel march; when there is no workspace (a first call under stream
capture); and the bounds on segments are reported for the same rays although a ray may be marched
beyond the sample that ends it."""
import numpy as np
import pytest

import synth
from synth.amr import random_hierarchy
from gpu_util import gpu_render, params_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amr():
    import paper_1212_3333_gb300 as m

    return m


def _hierarchy(seed=3):
    """1,629 leaves: the split march is for hierarchies of 1,000 and more."""
    return random_hierarchy(seed, n0=16, num_levels=4, patches_per_level=40, max_size=8)


def _context(amr, seed=3, maxbrick=True, gradient=True, storage="ptr", halo=2, dtype="f32"):
    h = _hierarchy(seed)
    ctx = amr.from_hierarchy(h, dtype)
    ctx.amr_build_kdtree(storage, gradient=gradient, halo=halo, maxbrick=maxbrick)
    return ctx, h.value_range()


def _opaque_tf(n=64, clear=16):
    """Opaque but for its first `clear` entries (none: the split march leaves every tile)."""
    tf = synth.ramp_tf(n)
    tf[:, 3] = 1.0
    tf[:clear, 3] = 0.0
    return tf


# samples per pixel from a few (one round) to far more than a tile may take (320 tasks per
# pixel)
@pytest.mark.parametrize("step", [0.5, 0.1, 0.01])
@pytest.mark.parametrize("size", [(33, 29), (160, 121)])
@pytest.mark.parametrize("maxbrick", [True, False])
def test_full_workspace_equals_per_ray(amr, step, size, maxbrick):
    ctx, (vmin, vmax) = _context(amr, maxbrick=maxbrick)
    cam = synth.orbit_camera(2, *size)
    for kappa, ert, clear in ((0.05, 0.0, 16), (3.0, 1e-3, 16), (0.05, 0.0, 0)):
        got = []
        for schedule in (0, 3):
            p, _ = params_pair(amr, vmin, vmax, schedule=schedule, shade=1, step_factor=step,
                               kappa=kappa, ert_eps=ert)
            got.append(gpu_render(ctx, cam, _opaque_tf(clear=clear), p))
        assert got[0][1] == got[1][1]
        assert np.array_equal(got[0][0], got[1][0])


@pytest.mark.parametrize("storage,dtype,maxbrick", [
    ("ptr", "f32", True), ("ptr", "f32", False), ("ptr", "f16", True), ("ptr", "bf16", False),
    ("atlas_linear", "f32", False), ("atlas_linear", "f16", False)])
@pytest.mark.parametrize("gradient,halo", [(True, 2), (True, 1), (False, 1)])
def test_storages_and_pruning_equal_per_ray(amr, storage, dtype, maxbrick, gradient, halo):
    ctx, (vmin, vmax) = _context(amr, 5, maxbrick, gradient, storage, halo, dtype)
    cam = synth.orbit_camera(9, 61, 50)
    for lod, skip, row0, rows in ((0.0, 0, 0, 0), (3.0, 0, 0, 0), (12.0, 0, 0, 0), (0.0, 1, 13, 21)):
        got = []
        for schedule in (0, 3):
            p, _ = params_pair(amr, vmin, vmax, schedule=schedule, shade=1, kappa=20.0,
                               lod_pixels=lod, skip=skip, row0=row0, rows=rows)
            got.append(gpu_render(ctx, cam, _opaque_tf(), p))
        assert got[0][1] == got[1][1] > 0
        assert np.array_equal(got[0][0], got[1][0])


@pytest.mark.parametrize("maxbrick", [True, False])
@pytest.mark.parametrize("shadow", [0, 1])
def test_small_workspace_takes_tiles_up_again(amr, monkeypatch, maxbrick, shadow):
    """256 chunks for 620 tiles of up to a chunk each (denser ones are left): some are given up and
    taken up again, with the second transfer function in two rounds and more, as a round has
    room for at most 256."""
    ctx, (vmin, vmax) = _context(amr, maxbrick=maxbrick)
    cam = synth.orbit_camera(2, 160, 121, fov_y_deg=18.0)
    tfs = [_opaque_tf(clear=20), _opaque_tf(clear=8)]
    want = []
    for tf in tfs:
        p, _ = params_pair(amr, vmin, vmax, schedule=0, shade=1, kappa=0.05, step_factor=8.0)
        if shadow:
            p.schedule = 3  # (images agree to rounding with the per-ray schedule's)
            p.shadow, p.light_step = 1, 0.02
            for a in range(3):
                p.light[a] = 0.4 + 0.1 * a
        want.append(gpu_render(ctx, cam, tf, p))
    small, _ = _context(amr, maxbrick=maxbrick)
    monkeypatch.setenv("AMR_FAULT", "small_pool")
    p.schedule = 3
    for tf, (img, n) in zip(tfs, want):
        got = gpu_render(small, cam, tf, p)
        assert got[1] == n and np.array_equal(got[0], img)
        tiles, left, again, dense = small.amr_get_task_counts()
        assert tiles >= 620 and again > (256 if tf is tfs[1] else 0) and dense > 0, (left, again)
    few, _ = _context(amr, maxbrick=maxbrick)
    monkeypatch.setenv("AMR_FAULT", "few_tiles")  # 20 tiles a row: three bands of 48 rows
    for tf, (img, n) in zip(tfs, want):
        got = gpu_render(few, cam, tf, p)
        assert got[1] == n and np.array_equal(got[0], img)
        assert 0 < few.amr_get_task_counts()[0] <= 240 + 2432


def test_segment_bound_is_reported_for_the_same_rays(amr):
    ctx, (vmin, vmax) = _context(amr)
    cam = synth.orbit_camera(5, 40, 31)
    seen = set()
    for kappa in (0.5, 400.0):  # the second ends every ray in its first segments
        for bound in (1, 2, 4, 64):
            got = []
            for schedule in (0, 3):
                p, _ = params_pair(amr, vmin, vmax, schedule=schedule, shade=1, kappa=kappa,
                                   ert_eps=0.2, max_segments=bound)
                try:
                    got.append(gpu_render(ctx, cam, _opaque_tf(clear=8), p))
                except amr.AmrError as e:
                    got.append(e.status)
            seen.add(isinstance(got[0], int))
            if isinstance(got[0], int):
                assert got[0] == got[1]
            else:
                assert got[0][1] == got[1][1] and np.array_equal(got[0][0], got[1][0])
    assert seen == {True, False}


# unshaded: hierarchies of 2,500 leaves and more through the split march up to 350,000 pixels,
# the others, and larger images, through the per-ray loop
@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("patches", [40, 100])
def test_unshaded_frames_equal_those_without_maximum_bricks(amr, dtype, patches):
    h = random_hierarchy(4, n0=16, num_levels=4, patches_per_level=patches, max_size=8)
    vmin, vmax = h.value_range()
    ctx = []
    for maxbrick in (False, True):
        ctx.append(amr.from_hierarchy(h, dtype))
        ctx[-1].amr_build_kdtree("ptr", halo=2, maxbrick=maxbrick)
    assert (ctx[0].amr_get_stats().num_leaves >= 2500) == (patches == 100)
    for size in ((67, 45), (700, 501)):
        for kappa, ert, clear, lod in ((0.5, 0.0, 40, 0.0), (0.5, 0.0, 0, 0.0), (40.0, 1e-3, 16, 0.0),
                                       (0.5, 0.0, 40, 3.0), (0.5, 0.0, 40, 12.0)):
            p, _ = params_pair(amr, vmin, vmax, schedule=0, shade=0, step_factor=0.3, kappa=kappa,
                               ert_eps=ert, lod_pixels=lod)
            cam = synth.orbit_camera(6, *size)
            (a, na), (b, nb) = (gpu_render(c, cam, _opaque_tf(clear=clear), p) for c in ctx)
            assert na == nb > 0 and np.array_equal(a, b)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("schedule", [0, -1])
def test_unshaded_frames_do_not_read_samples_per_iter(amr, dtype, schedule):
    """Schedule 0 takes any value of the field (it belongs to schedules 2 and 3)."""
    h = random_hierarchy(4, n0=16, num_levels=4, patches_per_level=100, max_size=8)
    ctx = amr.from_hierarchy(h, dtype)  # (3,000 leaves and more: the split march)
    ctx.amr_build_kdtree("ptr", halo=2, maxbrick=True)
    vmin, vmax = h.value_range()
    cam = synth.orbit_camera(2, 70, 53)
    want = None
    for spi in (16, 0, -1, 1, 65, 2 ** 31 - 1, -2 ** 31):
        p, _ = params_pair(amr, vmin, vmax, schedule=schedule, shade=0, step_factor=0.1,
                           samples_per_iter=spi)
        got = gpu_render(ctx, cam, _opaque_tf(), p)
        want = want or got
        assert got[1] == want[1] > 0 and np.array_equal(got[0], want[0]), spi


# the largest transfer functions whose shared memory, with the march kernels' static arrays,
# fits the default 48 KB, the first beyond it, those around 48 KB of their own, the longest
@pytest.mark.parametrize("shade", [0, 1])
@pytest.mark.parametrize("n", [1330, 1356, 1358, 1400, 1900, 1946, 2048])
def test_long_transfer_functions(amr, n, shade):
    ctx, (vmin, vmax) = _context(amr)
    plain, _ = _context(amr, maxbrick=False)
    cam = synth.orbit_camera(2, 40, 27)
    p, _ = params_pair(amr, vmin, vmax, schedule=0, shade=shade, step_factor=0.2)
    want = gpu_render(plain, cam, _opaque_tf(n, n // 4), p)
    for c in (ctx, plain):
        for schedule in (-1, 0, 2) + ((3,) if shade else ()):
            p.schedule = schedule
            got = gpu_render(c, cam, _opaque_tf(n, n // 4), p)
            assert got[1] == want[1] > 0 and np.array_equal(got[0], want[0]), schedule


def test_large_images_and_a_failing_launch(amr, monkeypatch):
    """Images of 3,000,000 pixels and more go through the split march on hierarchies of 10,000
    leaves and more, and leave what it does not take to the per-ray loop; a launch that fails
    before that is still reported."""
    from paper_1212_3333_gb300 import _lib

    h = random_hierarchy(7, n0=32, num_levels=4, patches_per_level=300, max_size=9)
    ctx = amr.from_hierarchy(h)
    ctx.amr_build_kdtree("ptr", gradient=True, halo=2, maxbrick=True)
    assert ctx.amr_get_stats().num_leaves >= 10000
    vmin, vmax = h.value_range()
    cam = synth.orbit_camera(4, 2003, 1501)
    # a few samples opaque, so many that the march stops on the way, all of them
    for clear, step in ((58, 0.5), (30, 0.1), (0, 0.5)):
        p, _ = params_pair(amr, vmin, vmax, schedule=0, shade=1, step_factor=step, kappa=0.01)
        want = gpu_render(ctx, cam, _opaque_tf(clear=clear), p)
        p.schedule = 3
        if clear:
            monkeypatch.setenv("AMR_FAULT", "shade_launch")
            with pytest.raises(amr.AmrError) as e:
                gpu_render(ctx, cam, _opaque_tf(clear=clear), p)
            assert e.value.status == _lib.AMR_ERR_CUDA
            monkeypatch.delenv("AMR_FAULT")
        got = gpu_render(ctx, cam, _opaque_tf(clear=clear), p)
        assert got[1] == want[1] and np.array_equal(got[0], want[0])


def test_first_call_captured(amr):
    import torch

    ctx, (vmin, vmax) = _context(amr)
    cam = synth.orbit_camera(7, 61, 47)
    tf = torch.as_tensor(_opaque_tf(), device="cuda")
    p, _ = params_pair(amr, vmin, vmax, schedule=3, shade=1)
    out = [torch.zeros((47, 61, 4), device="cuda") for _ in range(2)]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):  # no workspace yet, and none may be allocated
        ctx.amr_render(cam, tf, p, out[0])
    ctx.amr_render(cam, tf, p, out[1])
    g2 = torch.cuda.CUDAGraph()
    again = torch.zeros_like(out[0])
    with torch.cuda.graph(g2):  # with the workspace of the call before
        ctx.amr_render(cam, tf, p, again)
    big = torch.zeros((300, 400, 4), device="cuda")
    ctx.amr_render(synth.orbit_camera(8, 400, 300), tf, p, big)  # a larger workspace
    for graph in (g, g2):
        graph.replay()
    torch.cuda.synchronize()
    assert float(out[1].abs().max()) > 0
    assert torch.equal(out[0], out[1]) and torch.equal(again, out[1])


def test_one_workspace_at_a_time(amr):
    """Images of growing sizes replace the context's workspace; one that a captured call holds
    stays, and its replays give the same image; destroying the context gives all back."""
    import torch

    ctx, (vmin, vmax) = _context(amr)
    tf = torch.as_tensor(_opaque_tf(), device="cuda")
    p, _ = params_pair(amr, vmin, vmax, schedule=3, shade=1)
    outs = [torch.zeros((h, w, 4), device="cuda") for w, h in ((97, 61), (640, 479), (1700, 1000))]
    cams = [synth.orbit_camera(2, o.shape[1], o.shape[0]) for o in outs]
    first = torch.zeros_like(outs[0])
    torch.cuda.synchronize()
    free = [torch.cuda.mem_get_info()[0]]

    def render(k):
        ctx.amr_render(cams[k], tf, p, outs[k])
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])

    render(0)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.amr_render(cams[0], tf, p, first)
    for k in (1, 2, 1, 0, 2):
        render(k)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(first, outs[0])
    used = [(free[0] - f) / 1e9 for f in free]
    slack = used[1] + 0.1  # the captured call's workspace; the allocator's rounding
    assert 1.6 < used[2] < 1.8 + slack and 3.3 < used[3] < 3.6 + slack
    assert max(used[4:]) <= used[3] + 0.01
    del g
    ctx.amr_destroy()
    assert torch.cuda.mem_get_info()[0] >= free[0] - 10 ** 8


def test_calls_on_two_streams_take_turns(amr):
    """The streams share the context's workspace and counters: the second call waits for the
    first, so images and sample counts are those of calls made one at a time."""
    import torch

    ctx, (vmin, vmax) = _context(amr)
    cams = [synth.orbit_camera(s, 180, 150) for s in (1, 2, 3)]
    tf = torch.as_tensor(_opaque_tf(), device="cuda")
    ps = [params_pair(amr, vmin, vmax, schedule=schedule, shade=shade, step_factor=0.05, kappa=0.2)[0]
          for schedule, shade in ((3, 1), (3, 1), (0, 0))]
    want = []
    for cam, p in zip(cams, ps):
        out = torch.zeros((150, 180, 4), device="cuda")
        want.append((out, ctx.amr_render(cam, tf, p, out, count_samples=True)))
    streams = [torch.cuda.Stream() for _ in cams]
    got = [torch.zeros_like(w) for w, _ in want]
    torch.cuda.synchronize()
    for counted in (0, 1, 2, None):
        for k in range(6):
            i = (k + (counted or 0)) % 3
            n = ctx.amr_render(cams[i], tf, ps[i], got[i], stream=streams[i],
                               count_samples=i == counted)
            assert n is None or n == want[i][1]
    torch.cuda.synchronize()
    for g, (w, _) in zip(got, want):
        assert torch.equal(g, w)


def test_calls_on_streams_that_are_destroyed_take_turns(amr):
    """A new stream may get a destroyed one's handle while its work is still under way."""
    import ctypes

    import torch

    ctx, (vmin, vmax) = _context(amr)
    rt = torch.cuda.cudart()
    cam = synth.orbit_camera(1, 300, 250)
    tf = torch.as_tensor(_opaque_tf(), device="cuda")
    p, _ = params_pair(amr, vmin, vmax, schedule=3, shade=1, step_factor=0.05, kappa=0.2)
    outs = [torch.zeros((250, 300, 4), device="cuda") for _ in range(12)]
    ctx.amr_render(cam, tf, p, outs[0])
    torch.cuda.synchronize()
    for out in outs[1:]:
        h = ctypes.c_void_p()
        assert int(rt.cudaStreamCreate(ctypes.addressof(h))) == 0
        ctx.amr_render(cam, tf, p, out, stream=h.value)
        assert int(rt.cudaStreamDestroy(h.value)) == 0
    torch.cuda.synchronize()
    for out in outs[1:]:
        assert torch.equal(out, outs[0])
