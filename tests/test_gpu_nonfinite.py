"""Colours that overflow to infinity: the forward image is not finite exactly where they are
applied, and the gradients of Gaussians that share no pixel with one are what they are beside
ordinary colours.  Small images (every tile split over two blocks) and large ones (whole)."""
import numpy as np
import pytest

import oracle
from paper_2603_23891_gb300 import synth

from gpu_util import dev_params

pytestmark = pytest.mark.gpu

STEP = 4          # pixels between sites
DEEP = 3          # Gaussians of a site, one behind the other


def _scene(size):
    """Gaussians of half a pixel (0.45, 0.5 and 0.55 along their axes, turned about the line of
    sight) in the middle of every 4x4 pixels, a pixel off the blocks' grid, degree 3.  alpha0 =
    1/2 falls to 1/255 at 3.12 standard deviations of 0.71 to 0.78 pixels: the 4x4 pixels
    (farthest centre 2.12 pixels away), not their neighbours (2.55).  So sites share blocks,
    and the two pixels of a lane, but no pixels (a narrow view: perspective stretches a
    footprint by less than 2%, to 2.48 pixels).  Returns the hot nodes, one of every Gaussian
    of some sites, and the nodes of the other sites."""
    W, H = size
    cam = synth.look_at_camera([0, 0, 0], [0, 1, 0], W, H, 12.0)
    rng = np.random.default_rng(3)
    u, v = (np.repeat(x.ravel(), DEEP) for x in np.meshgrid(np.arange(3.0, W - 3, STEP), np.arange(3.0, H - 3, STEP)))
    n = len(u)
    z = rng.uniform(9.0, 11.0, n)
    R, t = np.asarray(cam.R, np.float64).reshape(3, 3), np.asarray(cam.t, np.float64)
    mu = (np.stack([(u - cam.cx) * z / cam.fx, (v - cam.cy) * z / cam.fy, z], 1) - t) @ R
    site = np.arange(n) // DEEP
    chosen = rng.random(n // DEEP) < 0.15
    hot = chosen[site] & (np.arange(n) % DEEP == rng.integers(0, DEEP, n // DEEP)[site])
    sh = rng.normal(0, 0.1, (n, 16, 3))
    sh[:, 0] += 1.0
    sh[:, 1, 0] = site                                     # (finds the site again in the tree's order)
    sh[:, 1, 1] = hot
    a = rng.uniform(0, np.pi, n)
    quat = np.stack([np.cos(a / 2), 0 * a, np.sin(a / 2), 0 * a], 1)
    scale = np.log(np.array([0.45, 0.5, 0.55]) * (z / cam.fx)[:, None])
    tree = synth.tree_from_gaussians(mu, scale, quat, np.zeros(n), sh, 3)
    leaf = np.asarray(tree.is_leaf) != 0
    of, is_hot = tree.sh[:, 1, 0].copy(), leaf & (tree.sh[:, 1, 1] == 1.0)
    tree.sh[:, 1] = 0.1
    apart = leaf & ~np.isin(of, of[is_hot])
    return tree, cam, np.nonzero(is_hot)[0], np.nonzero(apart)[0]


def _overflowing(sh, hot):
    """Coefficients whose terms all add up, to more than the largest binary32 value: the signs
    of the basis around (0, 1, 0)."""
    sh = np.array(sh, np.float32)
    signs = np.zeros(16, np.float32)
    for k, s in ((0, 1), (1, -1), (6, -1), (8, -1), (9, 1), (11, 1)):
        signs[k] = s
    sh[hot] = (3.0e38 * signs)[:, None]
    return sh


@pytest.mark.parametrize("size", [(96, 64), (1920, 1080)])
def test_infinite_colours(renderer, size):
    import torch
    tree, cam, hot, apart = _scene(size)
    renderer.load_tree(tree)
    renderer.set_params(tau_R=-1.0, tile=(16, 16), bg=(0.1, 0.2, 0.3))
    renderer.set_camera(cam)
    renderer.shrink(None)
    gp = oracle.GaussParams.of_tree(tree)
    params = dev_params(gp)
    dL = torch.rand(3, size[1], size[0], device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    moved = np.array(gp.sh)
    moved[hot] *= 0.5
    out = []
    for sh in (gp.sh, moved, _overflowing(gp.sh, hot)):
        params["sh"] = torch.from_numpy(np.ascontiguousarray(sh, np.float32)).cuda()
        renderer.update_params(params)
        rgb, T, _ = renderer.render(stats=True, keep=True)
        g = renderer.backward(dL, params)
        torch.cuda.synchronize()
        spl = renderer.splats()
        out.append((rgb.cpu(), T.cpu(), {k: v.cpu() for k, v in g.items()}, spl))
    (a, Ta, ga, _), (b, *_), (c, Tc, gc, spl) = out
    sel = renderer.filter()
    is_hot = np.isin(sel, hot)
    assert np.isinf(spl[is_hot][:, 8:11]).all() and np.isfinite(spl[~is_hot]).all()
    touched = (a != b).any(dim=0)
    assert touched.any() and not touched.all()
    assert torch.equal(~torch.isfinite(c).all(dim=0), touched)
    assert torch.equal(Ta, Tc) and torch.equal(a[:, ~touched], c[:, ~touched])
    for k in ga:
        x, y = ((v if k in ("logit", "sh") else v.t())[apart] for v in (ga[k], gc[k]))
        assert torch.isfinite(x).all()
        bad = ~torch.isfinite(y)
        assert not bad.any(), (k, int(bad.sum()))
        # the same products in another order of the blocks' reductions: 1e-4 of the largest
        # gradient is some 1,700 roundings of it
        assert float((x - y).abs().max()) <= 1e-4 * float(x.abs().max()), k
