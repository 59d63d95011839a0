"""Buckets in which most depths crowd together beside a few far ones (the sort then goes by
all bits of the depths from its first pass on) and buckets of tens of thousands of pairs,
for the three forms of the sort, against the oracle: pairs and values in order."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

from gpu_util import assert_frame_parity, gpu_frame, oracle_frame

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spread", [0.0, 1e-6, 1e-4, 1e-2])
@pytest.mark.parametrize("far", [0.0, 0.02, 0.5])
@pytest.mark.parametrize("counts", [[33, 40, 65, 100, 129, 256], [257, 513, 1025, 2048], [2049, 4000, 8191, 8192, 8193], [40000]])
def test_crowded(renderer, counts, far, spread):
    """All depths within a relative `spread` of 20, but for a share `far` of them anywhere
    between 1 and 40; a tenth exactly equal."""
    W, H = 16 * len(counts), 16
    cam = synth.look_at_camera([0.0, 0.0, 0.0], [0.0, 1.0, 0.0], W, H, 60.0)
    R, t = np.asarray(cam.R, np.float64).reshape(3, 3), np.asarray(cam.t, np.float64)
    rng = np.random.default_rng(29)
    pts = []
    for i, c in enumerate(counts):
        u, v = 16 * i + rng.uniform(5.0, 11.0, c), rng.uniform(5.0, 11.0, c)
        z = 20.0 * (1.0 + spread * rng.uniform(-1.0, 1.0, c))
        z = np.where(rng.random(c) < far, rng.uniform(1.0, 40.0, c), z)
        z[rng.integers(0, c, c // 10)] = 20.0
        pts.append((np.stack([(u - cam.cx) * z / cam.fx, (v - cam.cy) * z / cam.fy, z], 1) - t) @ R)
    mu = np.concatenate(pts)
    n = mu.shape[0]
    tree = synth.tree_from_gaussians(mu, np.full((n, 3), -7.0), np.tile([1.0, 0, 0, 0], (n, 1)),
                                     rng.normal(-3, 1, n), rng.normal(0, 1, (n, 1, 3)), 0)
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, -1.0)
    o, _ = oracle_frame(tree, cam, -1.0)
    assert np.array_equal(np.bincount((o.keys >> np.uint64(32)).astype(np.int64), minlength=len(counts)), counts)
    assert_frame_parity(g, o)
