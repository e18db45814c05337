"""Training steps of many fields, whose weight gradients run in turn instead of
beside the rest: the fused kernels against the network's FP32 mode on both sides
of that rule, with the tolerances of test_gpu_fno_fused.py, and passes queued
behind one another give the bits of one pass alone."""
import numpy as np
import pytest

from paper_1307_6703_gb300.workloads import network_groups, network_pack, network_weights
from test_gpu_fno_fused import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [24, 25, 64])
def test_many_fields(batch):
    import torch
    from paper_1307_6703_gb300.fno import Fno
    nx, ny, layers, mx, my = 32, 12, 2, 8, 4
    cfg = dict(width=32, hidden=64, layers=layers, modes_x=mx, modes_y=my, outputs=3)
    rng = np.random.default_rng(batch)
    p = network_weights(32, 64, layers, mx, my, 3, outputs=3)
    for k in list(p):
        if k in ("p", "q1", "q2") or k.startswith("w"):
            p[k] = 0.1 * rng.standard_normal(p[k].shape)
        if k.startswith("R"):
            p[k] = p[k] * 20.0
    flat = network_pack(p, layers)
    prm = np.stack([rng.uniform(0, 0.035, batch), rng.uniform(3e-4, 1e-3, batch), rng.choice([32.0, 64.0], batch),
                    rng.uniform(0.925, 0.96, batch)], axis=1)
    target = rng.uniform(-1, 1, (batch, 3, ny, nx))
    out, loss, g = _run(p, flat, prm, target, cfg, nx, ny, True)
    out32, loss32, g32 = _run(p, flat, prm, target, cfg, nx, ny, False)
    assert np.abs(out - out32).max() <= 3e-2 * np.abs(out32).max() and abs(loss - loss32) <= 1e-2 * loss32
    at = 0
    for k in network_groups(layers):
        a, b = g[at:at + p[k].size], g32[at:at + p[k].size]
        at += p[k].size
        assert np.abs(a - b).max() <= 8e-2 * np.abs(b).max(), k
        assert a @ b >= 0.99 * np.linalg.norm(a) * np.linalg.norm(b), k
    net = Fno(batch_max=batch, nx_max=nx, ny_max=ny, gemm_bf16=True, **cfg).set_params(flat)
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    o, d, t = torch.empty((batch, 3, ny, nx), dtype=torch.float32, device="cuda"), dev(prm), dev(target)
    for _ in range(5):
        net.forward(d, nx, ny, o)
        net.backward(t, want_loss=False)
    assert np.array_equal(net.get_grads().astype(np.float64), g)
    net.close()
