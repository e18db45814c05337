"""The network's fused layer and projection kernels (32 channels, 32 or 64
hidden) at the edges of their tiles -- 128 sites of one row: rows shorter
than a tile, one site group more than a tile, one and several rows, one field
-- against the FP64 reference (forward) and against the network's FP32 mode,
whose gradients are checked by finite differences elsewhere.  Tolerances are
those of the BF16 network (test_gpu_fno.py): 3e-2 of the output's scale; per
parameter group 8e-2 of the gradient's scale and a cosine of 0.99."""
import numpy as np
import pytest

from oracle import fno as ref
from paper_1307_6703_gb300.workloads import network_groups, network_pack, network_weights

pytestmark = pytest.mark.gpu


def _run(p, flat, prm, target, cfg, nx, ny, bf16):
    import torch
    from paper_1307_6703_gb300.fno import Fno
    net = Fno(batch_max=len(prm), nx_max=nx, ny_max=ny, gemm_bf16=bf16, **cfg).set_params(flat)
    out = torch.empty((len(prm), cfg["outputs"], ny, nx), dtype=torch.float32, device="cuda")
    net.forward(torch.tensor(prm, dtype=torch.float32, device="cuda"), nx, ny, out)
    loss = net.backward(torch.tensor(target, dtype=torch.float32, device="cuda"))
    g = net.get_grads()
    net.close()
    return out.cpu().numpy().astype(np.float64), loss, g.astype(np.float64)


@pytest.mark.parametrize("hidden,layers,mx,my,outputs,batch,nx,ny", [
    (64, 4, 16, 8, 3, 2, 128, 24),
    (64, 2, 16, 8, 3, 1, 136, 9),
    (64, 2, 32, 4, 4, 2, 72, 8),
    (32, 2, 8, 2, 1, 3, 264, 5),
    (32, 1, 16, 4, 3, 1, 32, 4),
])
def test_fused_kernels(hidden, layers, mx, my, outputs, batch, nx, ny):
    cfg = dict(width=32, hidden=hidden, layers=layers, modes_x=mx, modes_y=my, outputs=outputs)
    rng = np.random.default_rng(nx * 7 + ny)
    p = network_weights(32, hidden, layers, mx, my, 3, outputs=outputs)
    for k in list(p):
        if k in ("p", "q1", "q2") or k.startswith("w"):
            p[k] = 0.1 * rng.standard_normal(p[k].shape)
        if k.startswith("R"):
            p[k] = p[k] * 20.0
    flat = network_pack(p, layers)
    prm = np.stack([rng.uniform(0, 0.035, batch), rng.uniform(3e-4, 1e-3, batch), rng.choice([32.0, 64.0], batch),
                    rng.uniform(0.925, 0.96, batch)], axis=1)
    target = rng.uniform(-1, 1, (batch, outputs, ny, nx))
    out, loss, g = _run(p, flat, prm, target, cfg, nx, ny, True)
    out32, loss32, g32 = _run(p, flat, prm, target, cfg, nx, ny, False)
    exact = ref.forward(p, ref.features(prm.astype(np.float32), nx, ny), layers, mx, my)
    assert np.abs(out - exact).max() <= 3e-2 * np.abs(exact).max()
    assert abs(loss - np.mean((out - target) ** 2)) <= 1e-5 * loss
    at = 0
    for k in network_groups(layers):
        a, b = g[at:at + p[k].size], g32[at:at + p[k].size]
        at += p[k].size
        assert np.abs(a - b).max() <= 8e-2 * np.abs(b).max(), k
        assert a @ b >= 0.99 * np.linalg.norm(a) * np.linalg.norm(b), k
