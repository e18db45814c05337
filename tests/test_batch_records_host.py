"""Room for the records of a batch (host logic, on a CUDA runtime without a
GPU).  The tile with record r of a lattice writes 32 bytes at 32 r of the
lattice's record array, and a lattice is cut into other tiles in a batch than
alone: every record index of every launch must lie in the array that the launch
is given.  Lattices on both sides of a device full of 64-row tiles, both forms
of the relaxation, large lattices beside small ones, several device sizes."""
import ctypes as C
import json
import os
import sys

import pytest

from fake_cuda import Fake, host_call

FP32, BF16 = 1, 2
# (precision, tau, SMs, lattices)
CASES = {
    "one_4096x1600": (FP32, 1.0, 152, [(4096, 1600)]),
    "one_4096x1600_bf16": (BF16, 1.0, 152, [(4096, 1600)]),
    "one_65536x66": (FP32, 1.0, 152, [(65536, 66)]),
    "one_4096x1280_tau2": (FP32, 2.0, 152, [(4096, 1280)]),
    "one_4096x1216_tau2": (FP32, 2.0, 152, [(4096, 1216)]),
    "large_beside_small": (FP32, 1.0, 152, [(256, 64)] * 4 + [(4096, 1600)] + [(256, 64)] * 4),
    "two_large": (FP32, 1.0, 152, [(4096, 1600), (2048, 1600)]),
    "just_below_full": (FP32, 1.0, 152, [(4096, 1536)]),
    "well_above_full": (FP32, 1.0, 152, [(4096, 3072)]),
    "ordinary": (FP32, 1.0, 152, [(1024, 256), (512, 128), (128, 64)]),
    "smallest": (BF16, 2.0, 152, [(8, 8)]),
    "fewer_sms": (FP32, 1.0, 20, [(1024, 640)]),
    "one_sm": (FP32, 1.0, 1, [(64, 640), (256, 128)]),
}


def _fits(case, workdir):
    """[(launch, records, room)] of single and multi-step launches of the batch
    and of its instances alone, and of their sums."""
    prec, tau, sms, dims = CASES[case]
    fake = Fake(workdir)
    fake.rt.fake_sms(sms)
    import paper_1307_6703_gb300 as lbm
    ps = [lbm.lb_params(nx, ny, 1, prec, 0.375, 1 / 3, 0.3, 0.1, tau, 1e-4, 32.0, 0.0, 0.0, 0.3, 2.0, 0.0, None)
          for nx, ny in dims]
    out = []

    def records(addr, size):  # room of the record array named by a SweepArgs
        words = (C.c_uint64 * (size // 8)).from_address(addr)
        dev = [w for w in words if fake.room(w)]
        return fake.room(dev[3 if prec == FP32 else 5]) // 32  # sinx, fin(, fdin), fout(, fdev), partials, ...

    def on_launch(name, grid, args):
        def pointer(i):
            return C.cast(args[i], C.POINTER(C.c_void_p))[0]
        if "sweep_batch" in name:
            sa, n = pointer(1), 2 * len(dims)
            size = fake.room(sa) // n
            items = (C.c_int32 * (fake.room(pointer(0)) // 4)).from_address(pointer(0))
            top = [0] * len(dims)
            steps = 3 if "multi" in name else 1
            for j in range(grid[0] // steps):
                top[items[5 * j]] = max(top[items[5 * j]], items[5 * j + 3] + 1)
            out.extend((name, top[i // 2], records(sa + i * size, size)) for i in range(n))
        elif "sweep_step_kernel" in name:
            out.append((name, grid[0] * grid[1], records(args[2], 512)))
        elif "sweep_multi_kernel" in name:
            out.append((name, C.cast(args[5], C.POINTER(C.c_int32))[0], records(args[4], 512)))
        elif "reduce_cta" in name:
            out.append((name, C.cast(args[1], C.POINTER(C.c_int32))[0], fake.room(pointer(0)) // 32))

    b = lbm.Batch(ps)
    for v in b:
        v.init_noise(1, 1.0, 0.01)
    fake.on_launch = on_launch
    b.step(1)
    for v in b:
        v.reduce()
    b.step(3)
    for v in b:
        v.step(1)
        v.step(3)
    return out


@pytest.mark.parametrize("case", CASES)
def test_every_record_has_room(case, tmp_path):
    out = host_call(__file__, case, tmp_path)
    kinds = " ".join(name for name, _, _ in out)
    for k in ("sweep_batch_kernel", "sweep_batch_multi_kernel", "sweep_step_kernel", "sweep_multi_kernel", "reduce_cta"):
        assert k in kinds, k
    for name, need, room in out:
        assert 0 < need <= room, (name, need, room)


if __name__ == "__main__":
    os.makedirs(sys.argv[2], exist_ok=True)
    print(json.dumps(_fits(sys.argv[1], sys.argv[2])))
