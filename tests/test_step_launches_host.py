"""What lb_step enqueues (host logic, on a CUDA runtime without a GPU)."""
import ctypes as C
import json
import os
import sys

import pytest

from fake_cuda import STREAM, Fake, host_call


def _handle(lbm, nx, ny, prec=1, tau=1.0):
    h = lbm.lb_create(lbm.lb_params(nx, ny, 1, prec, 0.375, 1 / 3, 0.3, 0.1, tau, 1e-4, 32.0, 0.0, 0.0, 0.3, 2.0, 0.0,
                                    STREAM))
    lbm.lb_init(h, 0, 1, 1.0, 0.01)
    return h


def _single_step_sums(fake):
    """Device pointers of a single step's arguments."""
    import paper_1307_6703_gb300 as lbm
    out = []

    def on_launch(name, grid, args):
        words = (C.c_uint64 * 60).from_address(args[2])
        out.append(len({w for w in words if fake.room(w)}))
    for prec in (1, 2):
        h = _handle(lbm, 512, 256, prec)
        fake.on_launch = on_launch
        lbm.lb_step(h, 1)
        fake.on_launch = None
        fake.clear()
        lbm.lb_reduce(h, [0.0] * 3)
        out.append([n for n in ("reduce_cta", "reduce_pass1") if any(n in c for c in fake.names())])
    return out


def test_single_steps_leave_the_records_to_the_reduction(tmp_path):
    """sinx, the two states (and their 16-bit planes), records and error flag:
    no arrival counter and no sums, which the last tile would add up in one warp
    after the step; lb_reduce adds the records."""
    assert host_call(__file__, "_single_step_sums", tmp_path) == [5, ["reduce_cta"], 7, ["reduce_cta"]]


FORBIDDEN = ("cudaMalloc", "cudaFree", "cudaStreamSynchronize", "cudaMemcpy", "cudaMemset")


def _odd(fake):
    """Calls of the steps of lattices of odd widths: small, large, large without
    memory for the dependency lists, large inside a capture."""
    import paper_1307_6703_gb300 as lbm
    out = {}
    for what, nx, ny, room in (("small", 33, 33, 0), ("large", 1021, 509, 0), ("no_memory", 1021, 509, 1), ("capture", 1021, 509, 0)):
        p = lbm.lb_params(nx, ny, 1, 1, 0.375, 1 / 3, 0.3, 0.1, 1.0, 1e-4, 32.0, 0.0, 0.0, 0.3, 2.0, 0.0, STREAM)
        if room:  # the lists' size as a handle with memory asks for it, then a handle that gets less
            fake.clear()
            lbm.lb_create(p)
            lists = [c[2] for c in fake.calls if c[0] == "cudaMalloc"][-3]
            fake.rt.fake_fail_at(lists)
        h = lbm.lb_create(p)
        fake.rt.fake_fail_at(0)
        lbm.lb_init(h, 0, 1, 1.0, 0.01)
        fake.rt.fake_capturing(int(what == "capture"))
        fake.clear()
        lbm.lb_step(h, 5)
        lbm.lb_step(h, 3)
        fake.rt.fake_capturing(0)
        names = fake.names()
        out[what] = [sum("sweep_multi" in n for n in names), sum("sweep_step" in n for n in names),
                     [n for n in names if n in FORBIDDEN]]
    return out


def test_steps_of_odd_widths_only_enqueue(tmp_path):
    """[multi-step launches, single steps, calls that allocate or wait]"""
    out = host_call(__file__, "_odd", tmp_path)
    assert all(v[2] == [] for v in out.values()), out
    assert out["small"][:2] == [0, 8] and out["large"][:2] == [2, 0]
    assert out["no_memory"][:2] == [0, 8] and out["capture"][:2] == [0, 8]


def _state(fake):
    """Strided copies of a state read and set, with and without memory for the
    staging buffer."""
    import numpy as np
    import paper_1307_6703_gb300 as lbm
    out = []
    for prec, nx in ((1, 57), (1, 64), (2, 64)):
        for room in (True, False):
            h = _handle(lbm, nx, 32, prec)
            f = np.zeros(lbm.lb_get_state(h), dtype=np.uint8)
            fake.rt.fake_fail_at(0 if room else f.nbytes)
            fake.clear()
            lbm.lb_get_state(h, f)
            lbm.lb_set_state(h, f)
            fake.rt.fake_fail_at(0)
            out.append(fake.names().count("cudaMemcpy2DAsync"))
    return out


def test_states_are_copied_in_one_piece(tmp_path):
    assert host_call(__file__, "_state", tmp_path) == [0, 18] * 3


if __name__ == "__main__":
    os.makedirs(sys.argv[2], exist_ok=True)
    print(json.dumps(globals()[sys.argv[1]](Fake(sys.argv[2]))))
