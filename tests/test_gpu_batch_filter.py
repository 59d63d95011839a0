"""The batched form's R&L and Ancestor filters and its counted compaction, per view
against the oracle's serial traversal: several compaction tiles per view (and tiles that
hold the end of one view and the start of the next), trees deeper and shallower than the
16 levels read at once, more views than a 32-bit mask holds, and views that see nothing."""
import numpy as np
import pytest

from paper_2603_23891_gb300 import synth

from gpu_util import oracle_frame, orbit_cameras

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


def _views(tree, n, seed):
    cams = list(orbit_cameras(tree, n, (64, 48), seed, dist=(5, 60)))[:n]
    centre = tree.mu.mean(axis=1)
    # every fourth view looks away from the scene
    return [c if i % 4 != 3 else
            synth.look_at_camera(centre + 200.0, centre + 400.0, c.width, c.height, 40.0)
            for i, c in enumerate(cams)]


@pytest.mark.parametrize("n_leaves,branching,n_views", [(3, (2, 3), 1), (40000, (2, 8), 5), (30000, (1, 2), 4),
                                                        (9000, (2, 4), 33)])
def test_batch_selection(renderer, n_leaves, branching, n_views):
    import torch
    tree = synth.random_small_tree(31, n_leaves=n_leaves, branching=branching, extent=25.0, log_scale_mean=-1.0)
    assert (tree.depth > 16) == (branching == (1, 2))
    cams = _views(tree, n_views, 5)
    renderer.load_tree(tree)
    renderer.set_params(tau_R=3.0, tile=(16, 16))
    want = [oracle_frame(tree, c, 3.0, blend=False)[0].sel for c in cams]
    renderer.batch_setup(cams)
    for _ in range(2):
        renderer.render_batch()
        torch.cuda.synchronize()
        got = renderer.batch_frame()
        for v in range(n_views):
            assert np.array_equal(got[v]["sel"], want[v]), v
    assert n_views < 4 or (any(len(w) == 0 for w in want) and any(len(w) for w in want))
