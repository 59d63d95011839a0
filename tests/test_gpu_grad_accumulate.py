"""An accumulating backward adds in full binary32: what the buffers hold is kept to the bit
where the new gradient is zero, subnormal values too, on and off the 16-byte grid."""
import numpy as np
import pytest

import oracle
from paper_2603_23891_gb300 import synth

from gpu_util import dev_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_adding_zero_changes_nothing(renderer, degree, offset):
    import torch
    tree = synth.random_small_tree(50 + degree, n_leaves=500, branching=(2, 5), sh_degree=degree, extent=12.0)
    cam = synth.look_at_camera([20.0, 6.0, 4.0], tree.mu.mean(axis=1), 96, 64, 50.0)
    renderer.load_tree(tree)
    renderer.set_params(tau_R=4.0, tile=(16, 16))
    renderer.shrink(None)
    renderer.set_camera(cam)
    params = dev_params(oracle.GaussParams.of_tree(tree))
    renderer.update_params(params)
    _, _, st = renderer.render(stats=True)
    assert st.n_selected > 64
    held = torch.tensor([1e-40, -3e-42, 2e-38, 1.5, -1e30], device="cuda")
    grads, want = {}, {}
    for k in oracle.GRAD_FIELDS:
        flat = held.repeat(params[k].numel() // 5 + 2)[: params[k].numel() + offset].clone()
        grads[k] = flat[offset:].view(params[k].shape)
        want[k] = grads[k].clone()
    renderer.backward(torch.zeros(3, 64, 96, device="cuda"), params, grads, accumulate=True)
    torch.cuda.synchronize()
    for k in oracle.GRAD_FIELDS:
        assert np.array_equal(grads[k].cpu().numpy().view(np.uint32), want[k].cpu().numpy().view(np.uint32)), k
