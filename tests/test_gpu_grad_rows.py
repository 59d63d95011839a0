"""Which rows the backward writes: every gradient of a node outside the selection is zero
and none keeps what the buffer held, for every SH degree, node counts that end inside a
32-node word and buffers off the 16-byte grid; and an accumulating call adds to what is
there and leaves the other nodes' rows alone."""
import numpy as np
import pytest

import oracle
from paper_2603_23891_gb300 import synth

from gpu_util import dev_params

pytestmark = pytest.mark.gpu

NAMES = ("mu", "log_scale", "quat", "logit", "sh")


@pytest.fixture(scope="module")
def renderer():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_23891_gb300 import build, filtergs
    build.build()
    r = filtergs.Renderer(device=0)
    yield r
    r.close()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_rows_written(renderer, degree, offset):
    import torch
    tree = synth.random_small_tree(40 + degree, n_leaves=701 + degree, branching=(2, 5), sh_degree=degree, extent=12.0)
    n = tree.mu.shape[1]
    cam = synth.look_at_camera([20.0, 6.0, 4.0], tree.mu.mean(axis=1), 96, 64, 50.0)
    renderer.load_tree(tree)
    renderer.set_params(tau_R=4.0, tile=(16, 16))
    renderer.shrink(None)
    renderer.set_camera(cam)
    params = dev_params(oracle.GaussParams.of_tree(tree))
    renderer.update_params(params)
    renderer.render()
    sel = torch.from_numpy(renderer.filter().astype(np.int64)).cuda()
    renderer.render()
    out = torch.ones(n, dtype=torch.bool, device="cuda")
    out[sel] = False
    assert 32 < len(sel) < n - 32
    dL = torch.rand(3, 64, 96, device="cuda")

    def buffers(fill):
        g = {}
        for k in NAMES:
            flat = torch.full((params[k].numel() + offset,), fill, device="cuda")
            g[k] = flat[offset:].view(params[k].shape)
        return g

    node_axis = lambda k, x: x if k in ("logit", "sh") else x.t()
    fresh = buffers(float("nan"))
    renderer.backward(dL, params, fresh, accumulate=False)
    added = buffers(0.25)
    renderer.backward(dL, params, added, accumulate=True)
    torch.cuda.synchronize()
    for k in NAMES:
        f, a = node_axis(k, fresh[k]), node_axis(k, added[k])
        assert torch.isfinite(f).all(), k
        assert (f[out] == 0).all() and (f[sel] != 0).any(), k
        assert (a[out] == 0.25).all(), k
        # the two calls' sums differ by the order of the blend's reductions and the rounding of
        # 0.25 + g: 1e-4 of the largest gradient is some 1,700 roundings of it
        tol = 1e-4 * float(f.abs().max()) + 2.0 ** -24
        assert float((a[sel] - 0.25 - f[sel]).abs().max()) <= tol, k
