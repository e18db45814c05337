"""FP32 lattices of odd widths on both sides of a device full of tiles (below it
steps are launched one by one, above it many in one launch): steps in one call
and one by one give the same bits, and the sums are those of the state.  The
sums' bound: nine populations a site added in FP64 on both sides, in another
order: 2^-40 of the mass."""
import numpy as np
import pytest

from gpu_util import solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_FP32  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402


@pytest.mark.parametrize("nx,ny", [(9, 8), (33, 33), (4095, 16), (509, 256), (15, 3647), (15, 3650), (1021, 509)])
@pytest.mark.parametrize("tau", [1.0, 2.0])
def test_one_call_or_many(nx, ny, tau):
    w = C2(0.05).with_(nx=nx, ny=ny, tau=tau, A0=3e-4, lam=32.0)
    a = solver_for(w, LB_FP32).init_noise(3, 1.0, 0.01).step(7)
    b = solver_for(w, LB_FP32).init_noise(3, 1.0, 0.01)
    for _ in range(7):
        b.step(1)
    f = a.get_state()
    assert a.t == b.t == 7 and np.array_equal(f, b.get_state())
    rc, (m, _, _) = a.reduce()
    mass = f.sum(dtype=np.float64)
    assert rc == 0 and abs(m - mass) <= 2.0 ** -40 * mass
    a.close()
    b.close()
