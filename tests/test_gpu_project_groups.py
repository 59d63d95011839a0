"""The projection's groups of 32 entries that emit nothing, before, between and after groups
that do (their SH rows are not staged), in one turn of the grid and in several."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

from gpu_util import assert_frame_parity, gpu_frame, oracle_frame

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree,n", [(0, 700), (3, 700), (3, 130000)])
def test_groups_that_emit_nothing(renderer, degree, n):
    rng = np.random.default_rng(n)
    mu = np.stack([rng.uniform(-3, 3, n), rng.uniform(8, 12, n), rng.uniform(-2, 2, n)], 1)
    tree = synth.tree_from_gaussians(mu, rng.normal(-4.0, 0.5, (n, 3)), rng.normal(0, 1, (n, 4)), rng.normal(0, 1, n),
                                     rng.normal(0, 0.3, (n, (degree + 1) ** 2, 3)), degree)
    cam = synth.look_at_camera([0.0, 0.0, 0.0], [0.0, 1.0, 0.0], 200, 136, 70.0)
    leaf = np.nonzero(np.asarray(tree.is_leaf) != 0)[0]
    faint = (np.arange(len(leaf)) // 64) % 3 != 1          # two of three runs of 64 leaves, the first among them
    tree.opacity[leaf[faint]] = np.float32(0.01)           # below tau: nothing emitted
    tree.ln_opacity[leaf[faint]] = np.log(np.float32(0.01))
    shrink = (0.02, float(np.float32(np.log(0.02))))
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, -1.0, shrink=shrink)
    o, _ = oracle_frame(tree, cam, -1.0, shrink=shrink)
    emits = (o.rect[:, 1] > o.rect[:, 0]) & (o.rect[:, 3] > o.rect[:, 2])
    groups = emits[: len(emits) // 32 * 32].reshape(-1, 32).any(axis=1)
    assert groups.any() and not groups.all()
    assert_frame_parity(g, o)
    renderer.shrink(None)
