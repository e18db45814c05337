"""The fused backward pass computes its weight gradients beside the layers
below, with two buffers in turn for the layers' dz: one to three layers (each
parity of the buffers, and the last one in the buffer that the first layer's
result takes).  Passes queued one after the other without a host
synchronisation, and passes captured in a graph, give the bits of a pass on
its own."""
import numpy as np
import pytest

from paper_1307_6703_gb300.workloads import network_pack, network_weights

pytestmark = pytest.mark.gpu

NX, NY, B = 136, 64, 3


def _data():
    import torch
    rng = np.random.default_rng(11)
    prm = np.stack([rng.uniform(0, 0.035, B), rng.uniform(3e-4, 1e-3, B), rng.choice([32.0, 64.0], B),
                    rng.uniform(0.925, 0.96, B)], axis=1)
    targets = [torch.tensor(rng.uniform(-1, 1, (B, 3, NY, NX)), dtype=torch.float32, device="cuda") for _ in range(2)]
    return torch.tensor(prm, dtype=torch.float32, device="cuda"), targets


def _net(layers, stream=None):
    from paper_1307_6703_gb300.fno import Fno
    flat = network_pack(network_weights(32, 64, layers, 16, 8, 3, outputs=3), layers)
    return Fno(layers=layers, batch_max=B, nx_max=NX, ny_max=NY, stream=stream).set_params(flat)


@pytest.mark.parametrize("layers", [1, 2, 3])
def test_queued_and_captured_passes_give_the_bits_of_one_pass(layers):
    import torch
    prm, targets = _data()
    out = torch.empty((B, 3, NY, NX), dtype=torch.float32, device="cuda")
    want = []
    for t in targets:
        net = _net(layers)
        net.forward(prm, NX, NY, out)
        net.backward(t)
        want.append(net.get_grads())
        net.close()
    assert not np.array_equal(want[0], want[1])

    net = _net(layers)
    for k in (0, 1, 1, 0, 0, 1):
        net.forward(prm, NX, NY, out)
        net.backward(targets[k], want_loss=False)
    assert np.array_equal(net.get_grads(), want[1])
    net.backward(targets[0], want_loss=False)  # again from the same forward pass
    assert np.array_equal(net.get_grads(), want[0])
    net.close()

    st = torch.cuda.Stream()
    net = _net(layers, st.cuda_stream)
    net.forward(prm, NX, NY, out)
    net.backward(targets[1])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        net.forward(prm, NX, NY, out)
        net.backward(targets[0], want_loss=False)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(net.get_grads(), want[0])
    net.close()
