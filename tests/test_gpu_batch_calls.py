"""Batched calls that follow one another without a wait: each renders its own cameras, with
and without graph replay, for view counts on both sides of the camera block's sizes."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("n_views", [1, 16, 17])
def test_calls_without_a_wait(renderer, n_views, graph):
    import torch
    tree = synth.random_small_tree(11, n_leaves=4000, branching=(2, 6), sh_degree=1, extent=20.0, log_scale_mean=-0.9)
    renderer.load_tree(tree)
    renderer.set_params(tau_R=3.0, tile=(16, 16))
    renderer.shrink(None)
    centre = tree.mu.mean(axis=1).astype(np.float64)
    calls = [[synth.look_at_camera(centre + [40 - 7 * v, -50 + 9 * k, 25], centre, 96 + 16 * (v % 3), 64, 60.0)
              for v in range(n_views)] for k in range(5)]
    want = []
    for cams in calls:
        for cam in cams:
            renderer.set_camera(cam)
            want.append([x.clone() for x in renderer.render()[:2]])
    renderer.batch_setup(calls[0])
    renderer.render_batch(stats=True)
    n = int(renderer.batch_offsets[-1])
    rgb, T = torch.empty(3 * n, device="cuda"), torch.empty(n, device="cuda")
    torch.cuda.synchronize()
    got = []
    for cams in calls:
        renderer.batch_set_cameras(cams)
        views = renderer.render_batch(rgb, T, graph=graph)[3]
        got += [(a.clone(), b.clone()) for a, b in views]
    torch.cuda.synchronize()
    for (a, b), (wa, wb) in zip(got, want):
        assert torch.equal(a, wa) and torch.equal(b, wb)
