"""Which stream the library's own copies and clears run on (host logic, on a CUDA
runtime without a GPU).  A handle on a stream of the program's own -- which does
not wait for the default stream -- may use default-stream work only after having
waited for it."""
import json
import os
import sys

import pytest

from fake_cuda import STREAM, Fake, host_call

WRITES = ("cudaMemset", "cudaMemcpy", "cudaMemsetAsync", "cudaMemcpyAsync", "cudaMemcpy2DAsync")


def _unordered(calls):
    """Writes on another stream than STREAM that nothing waits for before the
    next launch on STREAM, or before the calls end."""
    out, open_ = [], []
    for name, stream, _, grid in calls:
        if name in WRITES and stream != STREAM and name != "cudaMemcpyAsync":
            open_.append(name)
        elif name == "cudaStreamSynchronize" and stream == 0:
            open_ = []
        elif grid and stream == STREAM:
            out, open_ = out + open_, []
    return out + open_


def _params(lbm, nx, ny, prec):
    return lbm.lb_params(nx, ny, 1, prec, 0.375, 1 / 3, 0.3, 0.1, 1.0, 1e-4, 32.0, 0.0, 0.0, 0.3, 2.0, 0.0, STREAM)


def _steps(fake):
    """Multi-step launches: the first of a handle, after a change of the tiling,
    of an odd width, and of a batch."""
    import paper_1307_6703_gb300 as lbm
    out = {}
    for what, nx, prec in (("fp32", 512, 1), ("bf16", 512, 2), ("odd", 509, 1)):
        h = lbm.lb_create(_params(lbm, nx, 256, prec))
        lbm.lb_init(h, 0, 1, 1.0, 0.01)
        fake.clear()
        lbm.lb_step(h, 5)
        lbm.lb_set_seg_h(h, 2)
        lbm.lb_step(h, 5)
        out[what] = _unordered(fake.calls)
    b = lbm.Batch([_params(lbm, 512, 256, 1)] * 2, stream=STREAM)
    for v in b:
        v.init_noise(1, 1.0, 0.01)
    fake.clear()
    b.step(3)
    b[0].set_seg_h(2)
    b.step(3)
    out["batch"] = _unordered(fake.calls)
    return out


def _create(fake):
    """New handles, until the call returns."""
    import paper_1307_6703_gb300 as lbm
    from paper_1307_6703_gb300 import fno
    out = {}
    for what, nx, prec in (("fp64", 33, 0), ("fp32", 64, 1), ("odd", 57, 1), ("bf16", 64, 2)):
        fake.clear()
        lbm.lb_create(_params(lbm, nx, 32, prec))
        out[what] = _unordered(fake.calls)
    fake.clear()
    lbm.Batch([_params(lbm, 64, 32, 1)] * 2, stream=STREAM)
    out["batch"] = _unordered(fake.calls)
    fake.clear()
    fno.Fno(nx_max=64, ny_max=32, stream=STREAM)
    out["network"] = _unordered(fake.calls)
    return out


def test_a_new_handle_is_cleared_when_its_call_returns(tmp_path):
    out = host_call(__file__, "_create", tmp_path)
    assert out == {k: [] for k in ("fp64", "fp32", "odd", "bf16", "batch", "network")}


def test_dependency_lists_are_filled_on_the_handles_stream(tmp_path):
    assert host_call(__file__, "_steps", tmp_path) == {"fp32": [], "bf16": [], "odd": [], "batch": []}


if __name__ == "__main__":
    os.makedirs(sys.argv[2], exist_ok=True)
    print(json.dumps(globals()[sys.argv[1]](Fake(sys.argv[2]))))
