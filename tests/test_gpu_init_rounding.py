"""Initial states of FP32 lattices are the FP64 equilibrium rounded once, whatever
the fields hold.  The FP64 reference here rounds a few times itself, 8 * 2^-53 of
the value and so 2^-26 of a float's last place: half of that place and 2^-26 of it.
Fields outside the kernel's bounds -- zero, tiny, huge, negative, infinite and not
a number -- against the same expression in numpy."""
import numpy as np
import pytest

from gpu_util import solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_FP32  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402

CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
T0 = 1 / 3


def _feq(n, u, v, T):
    with np.errstate(all="ignore"):
        uu, out = u * u + v * v, []
        for i in range(9):
            cu = CX[i] * u + CY[i] * v if CX[i] and CY[i] else (CX[i] * u if CX[i] else (CY[i] * v if CY[i] else np.zeros_like(n)))
            cc = CX[i] ** 2 + CY[i] ** 2
            t3 = (T - T0) * (cc - 2 * T0) / (2 * T0 * T0)
            out.append(W9[i] * n * (((1 + cu / T0) + (cu * cu - T0 * uu) / (2 * T0 * T0)) + t3))
        return np.stack(out)


@pytest.mark.parametrize("nx,ny", [(1600, 1500), (1601, 700)])
@pytest.mark.parametrize("moving", [False, True])
def test_every_population_is_rounded_once(nx, ny, moving):
    w = C2(0.05).with_(nx=nx, ny=ny, lam=32.0)
    r = np.random.default_rng(nx)
    n = 1 + 0.4 * r.uniform(-1, 1, (ny, nx))
    u, v = (0.1 * r.uniform(-1, 1, (2, ny, nx))) if moving else (None, None)
    s = solver_for(w, LB_FP32).init_fields(n, u, v)
    got, z = s.get_state().astype(np.float64), np.zeros_like(n)
    ref = _feq(n, z if u is None else u, z if v is None else v, w.T)
    assert np.all(np.abs(got - ref) <= (0.5 + 2.0 ** -26) * np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64))
    s.close()


def _same(got, ref):
    """Equal, both infinite alike or both no number; or a float next to the
    reference (which may sit near the middle of two)."""
    with np.errstate(all="ignore"):
        r = ref.astype(np.float32)
        close = np.abs(got.astype(np.float64) - ref) <= 0.51 * np.spacing(np.abs(r)).astype(np.float64)
    return np.all((got == r) | (np.isnan(got) & np.isnan(r)) | close)


@pytest.mark.parametrize("nx", [64, 57])
def test_fields_of_any_value(nx):
    ny = 12
    w = C2(0.05).with_(nx=nx, ny=ny, lam=32.0)
    odd = np.array([np.inf, -np.inf, np.nan, 0.0, 1e-30, 1e-39, 1e-42, 1e-300, 1e30, 1e300, 3.5e38, -1.0, 2.0, 1e-18, 1e18])
    r = np.random.default_rng(nx)
    base = lambda k: k * r.uniform(-1, 1, (ny, nx))  # noqa: E731
    n, z = 1 + base(0.3), np.zeros((ny, nx))
    n.ravel()[3 * np.arange(odd.size) + 7] = odd
    s = solver_for(w, LB_FP32).init_fields(n)
    assert _same(s.get_state(), _feq(n, z, z, w.T))
    s.close()
    vel = np.array([0.125, 0.13, -0.3, 0.577350269, 0.8164966, 1.0, 1e3, 1e10, 1e-20, 1e-40, 1e-300])
    n, u, v = 1 + base(0.3), base(0.1), base(0.1)
    u.ravel()[5 * np.arange(vel.size) + 3] = vel
    v.ravel()[7 * np.arange(vel.size) + 6] = -vel
    n.ravel()[11 * np.arange(odd.size) + 1] = odd
    s = solver_for(w, LB_FP32).init_fields(n, u, v)
    assert _same(s.get_state(), _feq(n, u, v, w.T))
    s.close()


def test_noise_of_any_amplitude():
    for rho, amp in ((1.0, 0.01), (0.0, 1e-25), (1e25, 1e20), (1.0, 1.0)):
        w = C2(0.05).with_(nx=64, ny=32, lam=32.0)
        s = solver_for(w, LB_FP32).init_noise(5, rho, amp)
        k = np.arange(w.nx * w.ny, dtype=np.uint64)
        with np.errstate(over="ignore"):
            q = np.uint64(5) + (k + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
            q = (q ^ (q >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            q = (q ^ (q >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            q = q ^ (q >> np.uint64(31))
        n = (rho + amp * (2 * ((q >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1)).reshape(w.ny, w.nx)
        z = np.zeros_like(n)
        assert _same(s.get_state(), _feq(n, z, z, w.T))
        s.close()
