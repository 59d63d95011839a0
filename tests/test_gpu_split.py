"""Which tiles the blend splits follows from the tiles with pairs: frames of even load around
the counts where the rule turns (3/5 of 912 resident blocks, and 912), with one tile of
many more pairs and without, equal the oracle bit for bit in T."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

from gpu_util import assert_frame_parity, gpu_frame, oracle_frame

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heavy", [0, 400])
@pytest.mark.parametrize("cols,rows", [(78, 7), (137, 4), (457, 1), (911, 1), (152, 6), (1000, 1)])
def test_even_frames(renderer, cols, rows, heavy):
    """Six Gaussians a pixel across in every tile, twelve in some (on both sides of a quarter
    above the mean), and `heavy` more in one."""
    W, H = 16 * cols, 16 * rows
    cam = synth.look_at_camera([0.0, 0.0, 0.0], [0.0, 1.0, 0.0], W, H, 60.0)
    rng = np.random.default_rng(cols)
    count = np.where(rng.random(cols * rows) < 0.3, 12, 6)
    count[cols * rows // 2] += heavy
    tile = np.repeat(np.arange(cols * rows), count)
    n = len(tile)
    u = 16 * (tile % cols) + rng.uniform(5, 11, n)
    v = 16 * (tile // cols) + rng.uniform(5, 11, n)
    z = rng.uniform(5.0, 40.0, n)
    R, t = np.asarray(cam.R, np.float64).reshape(3, 3), np.asarray(cam.t, np.float64)
    mu = (np.stack([(u - cam.cx) * z / cam.fx, (v - cam.cy) * z / cam.fy, z], 1) - t) @ R
    scale = np.log(z / cam.fx * 0.6)[:, None] + rng.uniform(-0.2, 0.2, (n, 3))
    tree = synth.tree_from_gaussians(mu, scale, np.tile([1.0, 0, 0, 0], (n, 1)), rng.normal(0, 1, n),
                                     rng.normal(0, 1, (n, 1, 3)), 0)
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, -1.0, bg=(0.1, 0.2, 0.3))
    o, _ = oracle_frame(tree, cam, -1.0, bg=(0.1, 0.2, 0.3))
    per_tile = np.bincount((o.keys >> np.uint64(32)).astype(np.int64), minlength=cols * rows)
    assert np.count_nonzero(per_tile) == cols * rows
    assert_frame_parity(g, o)
