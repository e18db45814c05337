"""A batch whose lattices fill the device alone: the batch cuts them into more
tiles than a solver of their own has, and each tile writes a record.  States
against a single solver's as tests/test_gpu_batch.py bounds them (2e-6 of the
largest population), sums of each instance against the FP64 sums of its state:
a record adds a column's at most 64 rows in FP32, so 65 roundings, 65 * 2^-24 of
the mass (momenta: of the sum of the magnitudes)."""
import numpy as np
import pytest

from gpu_util import rel_err, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_FP32, Batch  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402


@pytest.mark.parametrize("steps", [1, 3])
@pytest.mark.parametrize("tau,dims", [(1.0, [(4096, 1600)]), (2.0, [(4096, 1280)]),
                                      (1.0, [(256, 64), (4096, 1600), (128, 64)])], ids=["tau1", "tau2", "beside"])
def test_large_lattices_of_a_batch(tau, dims, steps):
    ws = [C2(0.05).with_(nx=nx, ny=ny, tau=tau, A0=3e-4, lam=32.0) for nx, ny in dims]
    alone = [solver_for(w, LB_FP32).init_noise(3, 1.0, 0.01) for w in ws]
    batch = Batch([s.params for s in alone])
    for v in batch:
        v.init_noise(3, 1.0, 0.01)
    batch.step(steps)
    for s, v in zip(alone, batch):
        s.step(steps)
        f = v.get_state()
        assert rel_err(f, s.get_state().astype(np.float64)) <= 2e-6
        rc, got = v.reduce()
        p = [f[i].sum(dtype=np.float64) for i in range(9)]
        tol = 65 * 2.0 ** -24 * sum(p)
        assert rc == 0 and abs(got[0] - sum(p)) <= tol
        assert abs(got[1] - (p[1] - p[3] + p[5] - p[6] - p[7] + p[8])) <= tol
        assert abs(got[2] - (p[2] - p[4] + p[5] + p[6] - p[7] - p[8])) <= tol
        # what lies behind the records is as it was: another step, same bounds
        s.step(1)
        v.step(1)
        assert rel_err(v.get_state(), s.get_state().astype(np.float64)) <= 2e-6
        s.close()
    batch.close()
