"""What a network holds on the device: one that is only evaluated, no more than its activations and two
layers' worth of gradients; its first gradients can be captured into a graph all the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _net(sizes, seed=0):
    from paper_2302_14344_gb300 import warmstart as ws
    rng = np.random.default_rng(seed)
    flat = [p for a, b in zip(sizes[:-1], sizes[1:])
            for p in (rng.standard_normal(a * b) * np.sqrt(2.0 / a), 0.1 * rng.standard_normal(b))]
    net = ws.Network(sizes)
    net.set_params(np.concatenate(flat).astype(np.float32))
    return net


def _data(sizes, batch):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    mk = lambda n: torch.randn((batch, n), generator=g, device="cuda")      # noqa: E731
    return mk(sizes[0]), mk(sizes[-1]), (mk(sizes[-1]) > 0).float()


def test_memory_of_an_evaluated_network():
    import torch
    sizes, batch = [64] + [256] * 12 + [16], 100000
    x, t, m = _data(sizes, batch)
    y = torch.empty_like(t)
    net = _net(sizes)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net.forward(x, y)
    torch.cuda.synchronize()
    held = free - torch.cuda.mem_get_info()[0]
    # BF16 inputs and FP32 pre-activations of every layer, FP32 outputs, two BF16 gradients; each
    # allocation is rounded up to at most 2 MB
    want = batch * (sum(2 * a + 4 * b for a, b in zip(sizes[:-1], sizes[1:])) + 4 * sizes[-1] + 2 * 2 * 256)
    assert held <= want + (2 * len(sizes) + 4) * (2 << 20), (held, want)


@pytest.mark.parametrize("sizes", [[32, 256, 256, 256, 7], [10, 33, 7], [5, 3], [8] + [24] * 10 + [4]])
def test_first_gradients_captured(sizes):
    """A graph of the gradients, captured after an evaluation only, and the direct call: equal up to the
    order of the batch's FP32 sums (2^-24 per term, 1000 terms: 1e-4 of the largest)."""
    import torch
    x, t, m = _data(sizes, 1000)
    net, ref = _net(sizes), _net(sizes)
    y = torch.empty_like(t)
    net.forward_layers(x, y)
    grad, want = (torch.zeros(net.num_params, device="cuda") for _ in range(2))
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    net.stream = st.cuda_stream
    with torch.cuda.graph(g, stream=st):
        net.gradients(x, t, m, grad)
    net.stream = 0
    g.replay()
    ref.gradients(x, t, m, want)
    torch.cuda.synchronize()
    assert float((grad - want).abs().max()) <= 1e-4 * float(want.abs().max())
    net.gradients(x, t, m, grad)                      # and the whole buffers from here on
    torch.cuda.synchronize()
    assert torch.equal(grad, want)
