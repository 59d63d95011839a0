"""The host side of the batched calls on a CPU: csrc/api.cu linked against replacements of
the CUDA runtime calls it makes and of the kernel launchers (fake_cuda.cpp,
fake_launchers.cu), driven through the binding's structs.  What the launches are given, in
which order host memory is read and rewritten, and what a failed call leaves; no kernel
runs."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def api(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    from paper_2603_23891_gb300 import build
    build.build()
    from paper_2603_23891_gb300 import filtergs
    so = str(tmp_path_factory.mktemp("host") / "libhost.so")
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-O1", f"-I{build.INCLUDE}", f"-I{build.CSRC}", "-Xcompiler", "-fPIC",
                    "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", so,
                    os.path.join(build.CSRC, "api.cu"), *(os.path.join(ROOT, "tests", f) for f in ("fake_launchers.cu", "fake_cuda.cpp"))],
                   check=True)
    L = C.CDLL(so)
    for name in filtergs.EXPORTED:
        if not hasattr(L, name):
            continue                                      # another file's entry point
        f, g = getattr(L, name), getattr(filtergs.lib(), name)
        f.argtypes, f.restype = g.argtypes, g.restype
    for name in ("fake_allocs", "fake_records", "fake_graphs", "fake_pinned", "fake_nulls"):
        getattr(L, name).restype = C.c_long
    L.fake_fail_at.argtypes = [C.c_long]
    L.fake_record.argtypes = [C.c_long, C.c_void_p, C.c_void_p, C.c_void_p]
    L.b = filtergs
    return L


@pytest.fixture
def ctx(api):
    h = C.c_void_p()
    assert api.fgs_create(C.byref(h), 0) == 0
    yield h
    api.fake_fail_at(-1)
    api.fgs_destroy(h)
    api.fake_clear()


def _load(api, ctx, n_leaves=200, seed=1):
    t = api.b._TreeArrays(synth.random_small_tree(seed, n_leaves=n_leaves, branching=(2, 5), sh_degree=1))
    assert api.fgs_load_tree(ctx, C.byref(t.struct)) == 0


def _cams(api, n, x):
    return api.b._cams([synth.look_at_camera([x + v, -30.0, 9.0], [x + v, 0, 0], 64, 48, 60.0) for v in range(n)])


def _setup(api, ctx, cams):
    return api.fgs_batch_setup(ctx, C.cast(cams, C.c_void_p), len(cams), None, 1 << 12, 1 << 12)


def _record(api, i):
    head, rgb, t = (C.c_int * 4)(), C.c_uint64(), np.zeros((64, 3), np.float32)
    api.fake_record(i, head, C.byref(rgb), t.ctypes.data)
    return dict(what=head[0], n_pad=head[2], nulls=head[3], rgb=rgb.value, t=t[:head[1]])


@pytest.mark.parametrize("flags", [0, 4])                  # 4: FGS_BATCH_GRAPH
@pytest.mark.parametrize("n_views", [1, 8, 17, 64])
def test_calls_in_flight_keep_their_cameras(api, ctx, n_views, flags):
    """Four batches enqueued without a wait between them, each with cameras and buffers of its
    own: every launch reads the cameras of its own call, however late it runs."""
    _load(api, ctx)
    assert _setup(api, ctx, _cams(api, n_views, 0.0)) == 0
    want = []
    for k in range(4):
        cams = _cams(api, n_views, 100.0 * k)
        want.append(np.array([list(c.t) for c in cams], np.float32))
        assert api.fgs_batch_set_cameras(ctx, C.cast(cams, C.c_void_p), n_views) == 0
        # with a graph the buffers stay: new ones capture again, which waits
        out = C.c_void_p(0x1000 if flags else 0x1000 * (k + 1))
        assert api.fgs_render_batch(ctx, None, out, out, flags, None) == 0
    api.fake_drain()
    recs = [_record(api, i) for i in range(api.fake_records())]
    assert [r["what"] for r in recs] == [0, 1] * 4
    for k in range(4):
        for r in recs[2 * k: 2 * k + 2]:
            assert r["nulls"] == 0 and np.array_equal(r["t"], want[k]), k


@pytest.mark.parametrize("flags", [0, 4])
def test_tree_loaded_after_the_set_up(api, ctx, flags):
    """A tree that the batch's buffers cannot hold is refused until the next set-up; one that
    they hold is rendered, and by a graph captured on that tree."""
    out = C.c_void_p(0x1000)
    _load(api, ctx, n_leaves=3000)                         # 4096 to 8192 nodes
    assert _setup(api, ctx, _cams(api, 3, 0.0)) == 0
    assert api.fgs_render_batch(ctx, None, out, out, flags, None) == 0
    assert api.fake_graphs() == (flags == 4)
    _load(api, ctx, n_leaves=30000)
    assert api.fake_graphs() == 0
    assert api.fgs_render_batch(ctx, None, out, out, flags, None) == api.b.FGS_ERR_STATE
    assert _setup(api, ctx, _cams(api, 3, 0.0)) == 0
    assert api.fgs_render_batch(ctx, None, out, out, flags, None) == 0
    _load(api, ctx, n_leaves=200)
    assert api.fake_graphs() == 0
    assert api.fgs_render_batch(ctx, None, out, out, flags, None) == 0
    api.fake_drain()
    n_pad = [_record(api, i)["n_pad"] for i in range(0, api.fake_records(), 2)]
    assert len(n_pad) == 3 and n_pad[0] > 4096 and n_pad[1] > n_pad[0] and n_pad[2] == 4096


@pytest.mark.parametrize("again", [False, True])
def test_failed_set_up_leaves_none(api, ctx, again):
    """Each allocation of the set-up fails in turn (the first set-up, or one that replaces
    another): the batch is refused afterwards, and the next set-up has every buffer."""
    out = C.c_void_p(0x1000)
    _load(api, ctx)
    for k in range(100):
        if again:
            assert _setup(api, ctx, _cams(api, 2, 0.0)) == 0
        api.fake_clear()
        api.fake_fail_at(k)
        cams = _cams(api, 5, 0.0)
        rc = api.fgs_batch_setup(ctx, C.cast(cams, C.c_void_p), 5, None, 1 << 13, 1 << 13)
        failed = api.fake_allocs() > k
        api.fake_fail_at(-1)
        assert rc == (api.b.FGS_ERR_NOMEM if failed else 0), k
        assert api.fgs_render_batch(ctx, None, out, out, 0, None) == (api.b.FGS_ERR_STATE if failed else 0), k
        api.fake_drain()
        assert api.fake_records() == (0 if failed else 2)
        if not failed:
            break
        assert _setup(api, ctx, _cams(api, 2, 0.0)) == 0
        assert api.fgs_render_batch(ctx, None, out, out, 0, None) == 0
        api.fake_drain()
        assert api.fake_records() == 2 and all(_record(api, i)["nulls"] == 0 for i in range(2)), k
    assert 12 <= k < 99


def test_refused_set_up_keeps_the_one_before(api, ctx):
    """A set-up with a wrong argument changes nothing."""
    out = C.c_void_p(0x1000)
    _load(api, ctx)
    assert _setup(api, ctx, _cams(api, 2, 0.0)) == 0
    cams = _cams(api, 5, 0.0)
    shapes = np.array([[16, 16, 8]] * 4 + [[16, 32, 8]], np.int32)
    for ts, cap in ((shapes.ctypes.data, 0), (None, 1 << 40)):
        assert api.fgs_batch_setup(ctx, C.cast(cams, C.c_void_p), 5, ts, 0, cap) == api.b.FGS_ERR_ARG
        assert api.fgs_render_batch(ctx, None, out, out, 0, None) == 0
    api.fake_drain()
    assert [len(_record(api, i)["t"]) for i in range(api.fake_records())] == [2] * 4


def test_failed_frame_buffers_are_not_used(api, ctx):
    """Each allocation of a growing pair list, image and tree fails in turn: frames are refused
    until the call is repeated, and no launch is given a null buffer."""
    rgb = C.c_void_p(0x1000)
    big = api.b._cams([synth.look_at_camera([0, -30.0, 9.0], [0, 0, 0], 640, 480, 60.0)])
    grow = {"pairs": lambda: api.fgs_set_params(ctx, C.byref(api.b.make_params(pair_capacity=1 << 14))),
            "camera": lambda: api.fgs_set_camera(ctx, big),
            "tiles": lambda: api.fgs_set_params(ctx, C.byref(api.b.make_params(tile=(64, 4)))),
            "tree": lambda: api.fgs_load_tree(ctx, C.byref(large.struct))}
    large = api.b._TreeArrays(synth.random_small_tree(1, n_leaves=9000, branching=(2, 5), sh_degree=1))
    nulls = api.fake_nulls()
    for name, call in grow.items():
        for k in range(100):
            h = C.c_void_p()
            api.fake_fail_at(-1)
            assert api.fgs_create(C.byref(h), 0) == 0
            ctx, keep = h, ctx
            _load(api, ctx)
            cam = api.b._cams([synth.look_at_camera([0, -30.0, 9.0], [0, 0, 0], 66, 48, 60.0)])
            assert api.fgs_set_camera(ctx, cam) == 0 and api.fgs_render(ctx, None, rgb, None, 1, 0, None) == 0
            api.fake_fail_at(k)
            rc = call()
            failed = api.fake_allocs() > k
            api.fake_fail_at(-1)
            assert rc == (api.b.FGS_ERR_NOMEM if failed else 0), (name, k)
            assert api.fgs_render(ctx, None, rgb, None, 1, 0, None) == (api.b.FGS_ERR_STATE if failed else 0), (name, k)
            assert call() == 0 and api.fgs_render(ctx, None, rgb, None, 1, 0, None) == 0
            if name != "tree":
                assert api.fgs_set_camera(ctx, cam) == 0
            else:
                _load(api, ctx)
            assert api.fgs_render(ctx, None, rgb, None, 1, 0, None) == 0
            assert api.fake_nulls() == nulls, (name, k)
            api.fgs_destroy(h)
            ctx = keep
            if not failed:
                break
        assert 0 < k < 99, name


def test_a_frame_needs_no_pinned_memory(api, ctx):
    """The calibration's pinned buffer is allocated by the first calibration, not by a camera
    of more tiles, and a failure leaves frames as they were."""
    rgb, gbar = C.c_void_p(0x1000), C.c_double()
    _load(api, ctx)
    small, large = (api.b._cams([synth.look_at_camera([0, -30.0, 9.0], [0, 0, 0], w, 48, 60.0)]) for w in (64, 640))
    pinned = api.fake_pinned()
    for cam in (small, large):
        assert api.fgs_set_camera(ctx, cam) == 0 and api.fgs_render(ctx, None, rgb, None, 1, 0, None) == 0
    assert api.fake_pinned() == pinned
    api.fake_fail_at(0)
    assert api.fgs_calibrate_view(ctx, None, C.byref(gbar), None, 0, None, 0) == api.b.FGS_ERR_NOMEM
    api.fake_fail_at(-1)
    assert api.fgs_render(ctx, None, rgb, None, 1, 0, None) == 0
    for cam in (small, large):
        assert api.fgs_set_camera(ctx, cam) == 0
        assert api.fgs_calibrate_view(ctx, None, C.byref(gbar), None, 0, None, 0) == 0
    assert api.fake_pinned() == pinned + 1


def _flat_tree(api, n):
    """A root and n - 1 leaves."""
    from types import SimpleNamespace
    parent = np.zeros(n, np.int32)
    parent[0] = -1
    ap = np.zeros((1, n), np.uint32)
    ap[0, 0] = 0xFFFFFFFF
    leaf = np.ones(n, np.uint8)
    leaf[0] = 0
    return api.b._TreeArrays(SimpleNamespace(
        mu=np.zeros((3, n)), cov=np.ones((6, n)), opacity=np.full(n, 0.5), ln_opacity=np.full(n, np.log(0.5)),
        sh=np.zeros((n, 1, 3)), sh_degree=0, parent=parent, is_leaf=leaf, ap=ap))


@pytest.mark.parametrize("first,then", [(2101248, 2097152), (2097152, 2093056), (2101248, 4096)])
def test_smaller_tree_with_the_same_set_up(api, ctx, first, then):
    """A set-up's bit arrays and counters hold every smaller tree's, 64 views of 2^22 words and
    fewer."""
    assert api.fgs_load_tree(ctx, C.byref(_flat_tree(api, first).struct)) == 0
    assert _setup(api, ctx, _cams(api, 64, 0.0)) == 0
    assert api.fgs_load_tree(ctx, C.byref(_flat_tree(api, then).struct)) == 0
    assert api.fgs_render_batch(ctx, None, C.c_void_p(0x1000), None, 0, None) == 0
    api.fake_drain()
    assert [_record(api, i)["nulls"] for i in range(api.fake_records())] == [0, 0]
