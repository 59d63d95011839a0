"""Trees whose ln_opacity does not describe their opacity (both are the caller's arrays): the
skip threshold comes from one and alpha from the other, so an applied alpha can be
subnormal, and a power below -87, where the blend's exp is 0, can pass the threshold."""
import numpy as np
import pytest

import oracle
from paper_2603_23891_gb300 import synth

from gpu_util import assert_frame_parity, gpu_frame, oracle_frame, orbit_cameras

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(96, 64), (1920, 1080)])
@pytest.mark.parametrize("opacity,ln_opacity", [(1e-38, 0.0), (1e-42, 0.0), (1e-12, 30.0), (0.5, 79.0), (0.5, 90.0), (1e-30, 130.0)])
def test_opacity_and_its_logarithm_apart(renderer, opacity, ln_opacity, size):
    tree = synth.random_small_tree(6, n_leaves=900, branching=(2, 6), sh_degree=0, extent=12.0, log_scale_mean=-2.0)
    odd = np.random.default_rng(1).random(tree.mu.shape[1]) < 0.3
    tree.opacity = np.where(odd, np.float32(opacity), tree.opacity).astype(np.float32)
    tree.ln_opacity = np.where(odd, np.float32(ln_opacity), tree.ln_opacity).astype(np.float32)
    cam = orbit_cameras(tree, 1, size, 4, dist=(14, 16), fov=(55, 60))[0]
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, 1.0, bg=(0.2, 0.3, 0.4))
    o, p = oracle_frame(tree, cam, 1.0, bg=(0.2, 0.3, 0.4))
    assert np.isin(np.nonzero(odd)[0], o.sel).sum() > 50
    assert_frame_parity(g, o)
    _, _, kpc = renderer.calibrate_view(want_kpc=True, n_pairs=len(o.keys))
    _, _, okpc = oracle.render(o.splat, o.keys, o.vals, cam, p, want_kpc=True)
    np.testing.assert_allclose(kpc, okpc, rtol=1e-4, atol=1e-5)     # test_gpu_parity.py's tolerance
