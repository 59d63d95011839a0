"""The batch's autotuning times each tile shape once a resolution class, and leaves the batch
set up with its choice, one of the candidates."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

pytestmark = pytest.mark.gpu


def test_each_shape_once(renderer, monkeypatch):
    import torch
    tree = synth.random_small_tree(3, n_leaves=500, branching=(2, 5), sh_degree=0, extent=12.0)
    renderer.load_tree(tree)
    renderer.set_params(tau_R=3.0, tile=(16, 16))
    centre = tree.mu.mean(axis=1)
    cams = [synth.look_at_camera([30.0, 10.0 * v, 20.0], centre, *((96, 64) if v % 2 else (64, 48)), 50.0) for v in range(4)]
    calls = []
    real = renderer.batch_setup
    monkeypatch.setattr(renderer, "batch_setup", lambda c, **k: (calls.append(k["tile_shapes"]), real(c, **k)))
    default = ((16, 16, 8), (16, 16, 4), (32, 8, 8), (32, 8, 4))
    choice, ms = renderer.batch_autotune(cams, sel_capacity=1 << 14, pair_capacity=1 << 18)
    assert len(calls) == 1 + 2 * 1 + 1 and ms > 0
    assert set(choice) == {(96, 64), (64, 48)} and set(choice.values()) <= set(default)
    calls.clear()
    shapes = ((32, 8, 4), (32, 8, 8), (16, 16, 8), (8, 32, 8), (16, 16, 4))
    choice, _ = renderer.batch_autotune(cams, candidates=shapes, sel_capacity=1 << 14, pair_capacity=1 << 18)
    assert len(calls) == 1 + 2 * 2 + 1 and set(choice.values()) <= set(shapes)
    assert [tuple(x) for x in calls[-1]] == [choice[(c.width, c.height)] for c in cams]
    want = []
    for cam in cams:
        tw, th, _ = choice[(cam.width, cam.height)]
        renderer.set_params(tile=(tw, th))
        renderer.set_camera(cam)
        want.append(renderer.render()[0].clone())
    views = renderer.render_batch(stats=True)[3]
    for (rgb, _), w in zip(views, want):
        assert np.array_equal(rgb.cpu().numpy(), w.cpu().numpy())
    torch.cuda.synchronize()
    renderer.set_params(tile=(16, 16))
