"""The projection's walk over the selection for every SH degree: a last group of 1 to 32
Gaussians, less than a block, and more Gaussians than the grid takes in one, two or three
turns, some emitting nothing; splat records, pairs and colours against the oracle."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

from gpu_util import assert_frame_parity, batch_view_frame, gpu_frame, oracle_frame

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


def _scene(n, degree):
    """n Gaussians in front of the camera, most of them small; one in eight is nearly
    transparent (it emits nothing when footprints are shrunk)."""
    rng = np.random.default_rng(100 + n)
    mu = np.stack([rng.uniform(-4, 4, n), rng.uniform(4, 12, n), rng.uniform(-3, 3, n)], 1)
    logit = rng.normal(0, 1, n)
    logit[::8] = -6.0
    K = (degree + 1) ** 2
    quat = rng.normal(0, 1, (n, 4))
    tree = synth.tree_from_gaussians(mu, rng.normal(-4.0, 0.5, (n, 3)), quat, logit, rng.normal(0, 0.3, (n, K, 3)), degree)
    return tree, synth.look_at_camera([0.0, 0.0, 0.0], [0.0, 1.0, 0.0], 200, 136, 70.0)


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 1000])
def test_small_selections(renderer, degree, n):
    tree, cam = _scene(n, degree)
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, -1.0, shrink=(0.02, float(np.float32(np.log(0.02)))))
    o, _ = oracle_frame(tree, cam, -1.0, shrink=(0.02, float(np.float32(np.log(0.02)))))
    assert_frame_parity(g, o)


@pytest.mark.parametrize("degree,n", [(3, 130000), (1, 260000), (2, 400000)])
def test_several_turns(renderer, degree, n):
    import torch
    tree, cam = _scene(n, degree)
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, -1.0)
    o, _ = oracle_frame(tree, cam, -1.0, blend=False)
    assert len(o.sel) > 100000
    assert_frame_parity(g, o, check_image=False)
    renderer.batch_setup([cam, cam])
    renderer.render_batch()
    torch.cuda.synchronize()
    for bv in renderer.batch_frame():
        assert_frame_parity(batch_view_frame(bv), o, check_image=False)
