"""Fields of more rows than a grid's y can count: forward and backward of the
fused kernels against the network's FP32 mode, with the tolerances of
test_gpu_fno_fused.py."""
import numpy as np
import pytest

from paper_1307_6703_gb300.workloads import network_groups, network_pack, network_weights
from test_gpu_fno_fused import _run

pytestmark = pytest.mark.gpu


def test_more_than_65535_rows():
    nx, ny, layers, mx, my = 16, 65600, 2, 8, 4
    cfg = dict(width=32, hidden=64, layers=layers, modes_x=mx, modes_y=my, outputs=1)
    rng = np.random.default_rng(5)
    p = network_weights(32, 64, layers, mx, my, 3, outputs=1)
    for k in list(p):
        if k in ("p", "q1", "q2") or k.startswith("w"):
            p[k] = 0.1 * rng.standard_normal(p[k].shape)
        if k.startswith("R"):
            p[k] = p[k] * 20.0
    flat, prm = network_pack(p, layers), np.array([[0.02, 5e-4, 32.0, 0.94]])
    target = rng.uniform(-1, 1, (1, 1, ny, nx))
    out, loss, g = _run(p, flat, prm, target, cfg, nx, ny, True)
    out32, loss32, g32 = _run(p, flat, prm, target, cfg, nx, ny, False)
    assert np.abs(out - out32).max() <= 3e-2 * np.abs(out32).max()
    assert abs(loss - loss32) <= 1e-2 * loss32
    at = 0
    for k in network_groups(layers):
        a, b = g[at:at + p[k].size], g32[at:at + p[k].size]
        at += p[k].size
        assert np.abs(a - b).max() <= 8e-2 * np.abs(b).max(), k
        assert a @ b >= 0.99 * np.linalg.norm(a) * np.linalg.norm(b), k
