"""The host side of the batched calls on a CPU: csrc/api.cu linked against replacements of
the CUDA runtime calls it makes and of the kernel launchers (fake_cuda.cpp,
fake_launchers.cu), driven through the binding's structs.  What the launches are given, in
which order host memory is read and rewritten; no kernel runs."""
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
    for name in ("fake_allocs", "fake_records", "fake_graphs", "fake_device_blocks"):
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
