"""The per-tile sort's passes over the depths' leading bits: buckets whose depths crowd
into a small part of their range, so that runs of equal leading bits are short (ordered
where they lie) or long (sorted again by every bit), in every size class, against the
oracle."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

from gpu_util import assert_frame_parity, gpu_frame, oracle_frame

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("crowd", [1.0, 1e-2, 1e-3, 1e-5, 0.0])
def test_crowded_depths(renderer, crowd):
    """One tile a bucket size; all depths but the nearest and the farthest within a relative
    `crowd` of one another, some of them equal.  At 16 leading bits of about 2^25 values of
    the range 5 to 40, 1e-2 leaves runs of a few, 1e-3 of tens, 1e-5 one run of all."""
    counts = [33, 64, 128, 200, 256, 257, 512, 700, 1024, 1500, 2048, 2049, 3000]
    W, H = 16 * len(counts), 16
    cam = synth.look_at_camera([0.0, 0.0, 0.0], [0.0, 1.0, 0.0], W, H, 60.0)
    R, t = np.asarray(cam.R, np.float64).reshape(3, 3), np.asarray(cam.t, np.float64)
    rng = np.random.default_rng(23)
    pts = []
    for i, c in enumerate(counts):
        u, v = 16 * i + rng.uniform(3.5, 12.5, c), rng.uniform(3.5, 12.5, c)
        z = 12.0 * (1.0 + crowd * rng.uniform(0.0, 1.0, c))
        z[rng.integers(0, c, c // 10)] = z[0]
        z[:2] = 5.0, 40.0
        pts.append((np.stack([(u - cam.cx) * z / cam.fx, (v - cam.cy) * z / cam.fy, z], 1) - t) @ R)
    mu = np.concatenate(pts)
    n = mu.shape[0]
    tree = synth.tree_from_gaussians(mu, np.full((n, 3), -6.0), np.tile([1.0, 0, 0, 0], (n, 1)),
                                     rng.normal(0, 1, n), rng.normal(0, 1, (n, 1, 3)), 0)
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, -1.0)
    o, _ = oracle_frame(tree, cam, -1.0)
    assert np.array_equal(np.bincount((o.keys >> np.uint64(32)).astype(np.int64), minlength=len(counts)), counts)
    assert_frame_parity(g, o)
