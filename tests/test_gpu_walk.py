"""The blend's walk at the edges of its groups, windows and chunks, in both forms (a
tile walked by one CTA, a tile split over two), against the oracle; and colours that
are not finite."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

from gpu_util import assert_frame_parity, gpu_frame, grad_parity_case, oracle_frame

pytestmark = pytest.mark.gpu

SPLIT = 912      # a tile with more than 1 / 912 of the frame's pairs is split


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


@pytest.mark.parametrize("whole", [False, True])
@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32), (64, 4)])
def test_list_lengths(renderer, tile, whole):
    """A row of tiles with 1 ... 260 overlapping low-opacity Gaussians of a few pixels each
    (around the group of 8 or 16, the window of two groups and the chunk of 128), alone
    (every tile split) and beside one tile of 240,000 opaque ones (most others whole)."""
    counts = [1, 7, 8, 9, 15, 16, 17, 32, 33, 64, 127, 128, 129, 136, 137, 255, 256, 257]
    rng = np.random.default_rng(5)
    cols = len(counts) + 2                                # an empty column before the filler's
    W, H = tile[0] * cols, tile[1]
    cam = synth.look_at_camera([0.0, 0.0, 0.0], [0.0, 1.0, 0.0], W, H, 60.0)
    R, t = np.asarray(cam.R, np.float64).reshape(3, 3), np.asarray(cam.t, np.float64)
    pts, scale, logit = [], [], []
    for i, c in enumerate(counts + [0] + ([240_000] if whole else [])):
        u = tile[0] * i + rng.uniform(3.0, tile[0] - 3.0, c)
        v = rng.uniform(min(3.0, tile[1] / 2), max(tile[1] - 3.0, tile[1] / 2), c)
        z = rng.uniform(5.0, 40.0, c)
        pts.append((np.stack([(u - cam.cx) * z / cam.fx, (v - cam.cy) * z / cam.fy, z], 1) - t) @ R)
        filler = i > len(counts)
        scale.append(np.log(z / cam.fx * (0.3 if filler else 1.2))[:, None] + rng.uniform(-0.5, 0.3, (c, 3)))
        logit.append(rng.normal(3.0 if filler else -2.0, 0.5, c))
    mu, scale, logit = (np.concatenate(x) for x in (pts, scale, logit))
    n = len(mu)
    quat = rng.normal(size=(n, 4))
    tree = synth.tree_from_gaussians(mu, scale, quat / np.linalg.norm(quat, axis=1, keepdims=True), logit,
                                     rng.normal(0, 1, (n, 1, 3)), 0)
    renderer.load_tree(tree)
    g = gpu_frame(renderer, tree, cam, -1.0, tile=tile)
    o, _ = oracle_frame(tree, cam, -1.0, tile=tile)
    per_tile = np.bincount((o.keys >> np.uint64(32)).astype(np.int64), minlength=cols)[:len(counts)]
    above = per_tile > len(o.keys) // SPLIT
    assert np.count_nonzero(above != whole) >= 9, above
    assert_frame_parity(g, o)


@pytest.mark.parametrize("size", [(96, 64), (1920, 1080)])
def test_infinite_colour_stays_where_it_is_applied(renderer, size):
    """One Gaussian's colour overflows: exactly the pixels that apply it are not finite,
    the others and every T keep their bits (96x64: split tiles; 1080p: whole ones)."""
    import torch
    rng = np.random.default_rng(8)
    wide, n = 20, 120
    mu = np.stack([rng.uniform(-6, 6, n), rng.uniform(10, 14, n), rng.uniform(-4, 4, n)], 1)
    logs = np.full((n, 3), -1.5)
    mu[:wide], logs[:wide] = [0.0, 12.0, 0.0], 2.5       # seen by every tile
    sh = rng.uniform(0.1, 1.0, (n, 1, 3))
    cam = synth.look_at_camera([0, 0, 0], [0, 1, 0], *size, 70.0)
    images = []
    for colour in (0.5, 1.5, 1e39):
        sh[60] = min(colour, 3e38)
        with np.errstate(over="ignore"):
            tree = synth.tree_from_gaussians(mu, logs, np.tile([1.0, 0, 0, 0], (n, 1)), np.full(n, -2.0), sh, 0)
        tree.sh[np.nonzero(np.isclose(tree.sh[:, 0, 0], np.float32(sh[60, 0, 0])))[0]] = min(colour, 3e38)
        if colour > 1e38:
            tree.sh[0] = 0.5                              # the root is not selected
        renderer.load_tree(tree)
        renderer.set_params(tau_R=-1.0, tile=(16, 16), bg=(0.1, 0.2, 0.3))
        renderer.set_camera(cam)
        renderer.shrink(None)
        rgb, T, _ = renderer.render(stats=True)
        torch.cuda.synchronize()
        images.append((rgb.cpu().numpy(), T.cpu().numpy()))
    (a, Ta), (b, Tb), (c, Tc) = images
    touched = (a != b).any(axis=0)
    assert touched.any() and not touched.all()
    assert np.array_equal(Ta.view(np.uint32), Tc.view(np.uint32))
    big = np.abs(c).max(axis=0) > 1e30
    assert np.array_equal(big | ~np.isfinite(c).all(axis=0), touched)
    assert np.array_equal(a[:, ~touched].view(np.uint32), c[:, ~touched].view(np.uint32))


@pytest.mark.parametrize("size", [(90, 70), (1920, 1080)])
@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32), (64, 4)])
def test_gradients_on_every_tile_shape(renderer, tile, size):
    """The gradient walk on a scene with tiles of up to hundreds of pairs, opaque enough
    that pixels stop inside the lists, against the oracle: split tiles (small image, every
    pixel), whole ones (1080p, a thousand pixels)."""
    rng = np.random.default_rng(12)
    n = 400
    mu = np.stack([rng.uniform(-7, 7, n), rng.uniform(8, 14, n), rng.uniform(-5, 5, n)], 1)
    logs = rng.uniform(-1.5, 0.8, (n, 3))
    quat = rng.normal(size=(n, 4))
    sh = rng.normal(0, 0.1, (n, 4, 3))
    tree = synth.tree_from_gaussians(mu, logs, quat / np.linalg.norm(quat, axis=1, keepdims=True),
                                     rng.normal(0.0, 1.5, n), sh, 1)
    cam = synth.look_at_camera([0, 0, 0], [0, 1, 0], *size, 70.0)
    small = size[0] < 1000
    pix = None if small else np.sort(rng.choice(size[0] * size[1], 1000, replace=False))
    g, _, _ = grad_parity_case(renderer, tree, cam, -1.0, 3, tile=tile, pix=pix)
    split = np.bincount((g["keys"] >> np.uint64(32)).astype(np.int64)) > g["NP"] // SPLIT
    assert split.all() if small else np.count_nonzero(~split) > 5000
