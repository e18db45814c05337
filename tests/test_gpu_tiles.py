"""The strip sweep at the edges of its tiles: a warp's tile is at most 56
columns wide (a 64-column window, two columns per lane) and a multiple of 2
or 4 rows high, and relaxation time 1 has a form of its own (no populations
in the collision).  Lattices one column quantum below, at and above one and
two tiles, heights around the tile heights, walls and periodic rows, tau = 1
and tau = 2, against the FP64 oracle; and the same lattice cut in different
ways, bit for bit.

Tolerance: a step rounds each population about 25 times (relative 2^-24
each), so five steps stay below 5 * 25 * 6e-8 = 7.5e-6 of the largest
population even if every rounding went the same way."""
import numpy as np
import pytest

from gpu_util import oracle_for, rel_err, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_FP32, Batch, lb_set_tiling  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402

STEPS, TOL = 5, 5 * 25 * 2.0 ** -24


def _w(nx, ny, walls, tau):
    u = 0.04 if walls else 0.0
    return C2(0.05).with_(nx=nx, ny=ny, walls=walls, tau=tau, A0=3e-4, lam=32.0, u_bot=-u, u_top=u)


def _n0(nx, ny):
    rng = np.random.default_rng(nx * 1000 + ny)
    y, x = np.mgrid[0:ny, 0:nx]
    return 1.0 + 0.3 * np.sin(2 * np.pi * y / ny) * np.cos(2 * np.pi * x / nx) + 0.01 * rng.uniform(-1, 1, (ny, nx))


@pytest.mark.parametrize("tau", [1.0, 2.0])
@pytest.mark.parametrize("walls", [True, False], ids=["walls", "periodic"])
@pytest.mark.parametrize("nx,ny", [(8, 8), (52, 9), (56, 10), (60, 11), (112, 13), (116, 33), (300, 67)])
def test_tile_edges_against_the_oracle(nx, ny, walls, tau):
    w = _w(nx, ny, walls, tau)
    n0 = _n0(nx, ny)
    s = solver_for(w, LB_FP32).init_fields(n0).step(STEPS)
    ref = oracle_for(w).init_fields(n0).step(STEPS)
    f = s.get_state()
    assert rel_err(f, ref.f) <= TOL
    # one launch per step, and other tilings: the same bits
    one = solver_for(w, LB_FP32).init_fields(n0)
    for _ in range(STEPS):
        one.step(1)
    assert np.array_equal(one.get_state(), f)
    for strips in {-(-nx // 116), -(-nx // 56), nx // 8}:
        for seg in (1, 2, 3, 4, 7, 64):
            t = solver_for(w, LB_FP32).init_fields(n0)
            lb_set_tiling(t.h, max(strips, -(-nx // 116)), seg)
            assert np.array_equal(t.step(STEPS).get_state(), f), (strips, seg)
            t.close()
    one.close()
    s.close()


@pytest.mark.parametrize("taus", [(1.0, 1.0, 1.0), (1.0, 2.0, 1.0)], ids=["tau1", "mixed"])
def test_batch_takes_the_form_of_all_its_lattices(taus):
    """A batch runs the tau = 1 form only when every lattice has tau = 1."""
    ws = [_w(56, 10, True, taus[0]), _w(120, 33, False, taus[1]), _w(64, 20, True, taus[2])]
    b = Batch([solver_for(w, LB_FP32).params for w in ws])
    n0 = [_n0(w.nx, w.ny) for w in ws]
    for v, n in zip(b, n0):
        v.init_fields(n)
    b.step(1).step(STEPS - 1)
    for v, w, n in zip(b, ws, n0):
        assert rel_err(v.get_state(), oracle_for(w).init_fields(n).step(STEPS).f) <= TOL
    b.close()


@pytest.mark.parametrize("walls", [True, False], ids=["walls", "periodic"])
@pytest.mark.parametrize("nx,ny", [(31, 3), (33, 4), (32, 15), (64, 16), (65, 17), (97, 61)])
def test_fp64_tiles_give_the_oracle_bit_for_bit(nx, ny, walls):
    """The FP64 tile kernel (32 columns by 4 to 16 rows, chosen by the lattice):
    one column or row below, at and above a tile, with velocities given."""
    from paper_1307_6703_gb300 import LB_FP64
    w = _w(nx, ny, walls, 2.0)
    rng = np.random.default_rng(nx + ny)
    f = [_n0(nx, ny), 0.05 * rng.uniform(-1, 1, (ny, nx)), 0.05 * rng.uniform(-1, 1, (ny, nx))]
    s = solver_for(w, LB_FP64).init_fields(*f).step(3)
    ref = oracle_for(w).init_fields(*f).step(3)
    assert np.array_equal(s.get_state(), ref.f)
    for g, r in zip(s.moments(), ref.moments()):
        assert np.array_equal(g, r)
