"""Gradients of networks whose widths and batches are not whole tiles (64 x 64 x 32), against
the FP64 reference that rounds to BF16 where the kernels store BF16.  Tolerance: the stored
activations and gradients carry one BF16 rounding (2^-9 relative) per layer, and a value that
falls on the other side of a rounding boundary moves by 2^-8: 5e-3 of an array's norm."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


# widths not a multiple of 8 take the element-wise copies, the others the 16-byte ones;
# batches around one split (128 rows), one K step and many splits of unequal length
@pytest.mark.parametrize("sizes", [[32, 256, 256, 256, 7], [5, 33, 70, 3], [8, 64, 72, 1]])
@pytest.mark.parametrize("B", [1, 31, 129, 1000, 2081])
def test_gradients_of_ragged_shapes(sizes, B):
    import torch
    from paper_2302_14344_gb300 import warmstart as ws
    rng = np.random.default_rng(B)
    params = [(W.astype(np.float32).astype(np.float64),
               (rng.standard_normal(b.shape) * 0.1).astype(np.float32).astype(np.float64))
              for W, b in mlp.init_params(sizes, seed=3)]
    x = rng.standard_normal((B, sizes[0])).astype(np.float32)
    t = rng.standard_normal((B, sizes[-1])).astype(np.float32)
    mask = (rng.random((B, sizes[-1])) < 0.85).astype(np.float32)
    net = ws.Network(sizes)
    net.set_params(ws.join_params(params))
    grad = torch.full((net.num_params,), float("nan"), device="cuda")
    d = lambda a: torch.from_numpy(a).cuda()
    net.gradients(d(x), d(t), d(mask), grad)
    y, cache = mlp.forward(params, x.astype(np.float64), bf16=True)
    ref = mlp.backward(params, cache, y, t.astype(np.float64), mask.astype(np.float64), bf16=True)
    for (gw, gb), (rw, rb) in zip(ws.split_params(grad.cpu().numpy().astype(np.float64), sizes), ref):
        assert np.linalg.norm(gw - rw) <= 5e-3 * np.linalg.norm(rw) + 1e-9
        assert np.linalg.norm(gb - rb) <= 5e-3 * np.linalg.norm(rb) + 1e-9
