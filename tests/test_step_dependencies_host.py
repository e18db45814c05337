"""The dependency lists that multi-step launches are given (host logic, on a CUDA
runtime without a GPU), against the boxes their copies read.

A tile of columns x0 .. x0 + W - 1 and rows ya .. yb - 1 reads the columns of its
TMA box (its width is in the descriptor) from x0 - 4 and rows ya - 4 .. yb + 4.  A
position is written by the tile that owns its site, or, for a ghost column or,
without walls, a ghost row, by the tile that owns the site it is an image of; with
walls the rows outside the lattice are never written, and neither are the columns
beyond the ghost band of four.  Every writer of a position a tile reads must be in
its list (it must have finished the step before), and the tile in every such
writer's (which must not overwrite what the tile has yet to read)."""
import ctypes as C
import json
import os
import struct
import sys

import pytest

from fake_cuda import Fake, host_call

FP32, BF16, FP16 = 1, 2, 3
# precision, tau, nx, ny, walls, SMs, segment height (None: the library's)
CASES = {
    "headline": (FP32, 1.0, 4096, 1024, 1, 152, None),
    "tuned": (FP32, 1.0, 4096, 1024, 1, 152, 52),
    "bf16": (BF16, 1.0, 1024, 256, 1, 152, None),
    "fp16_periodic": (FP16, 2.0, 2048, 512, 0, 152, None),
    "low_tiles": (FP32, 1.0, 512, 256, 0, 152, None),
    "one_row_tiles": (FP32, 2.0, 300, 130, 0, 152, 1),
    "smallest": (FP32, 1.0, 8, 8, 0, 1, None),
    "smallest_bf16": (BF16, 2.0, 8, 9, 1, 152, 3),
    "two_tiles": (FP32, 1.0, 64, 32, 0, 1, 5),
    "flat": (BF16, 1.0, 4096, 8, 0, 152, None),
    "odd_57": (FP32, 1.0, 57, 40, 0, 1, None),
    "odd_113": (FP32, 2.0, 113, 33, 1, 1, None),
    "odd_9": (FP32, 1.0, 9, 200, 0, 1, None),
    "odd_ragged": (FP32, 1.0, 1021, 509, 1, 152, None),
    "odd_narrow_last": (FP32, 1.0, 225, 61, 0, 1, None),
}


def _tiles(a):
    """Geometry of a SweepArgs: nx, ny, walls, seg_h, nseg, nstrips, base_w, extra, pad."""
    nx, ny, walls = struct.unpack_from("<3i", a, 0)
    return (nx, ny, walls) + struct.unpack_from("<6i", a, 32)


def _missing(geo, quantum, window, ofs, idx):
    """Entries that the lists lack, of (tile, writer) and (writer, tile)."""
    nx, ny, walls, seg_h, nseg, ncol, base, extra, pad = geo
    x0 = [i * base + quantum * min(i, extra) for i in range(ncol)] + [nx]
    assert all(0 < b - a <= window - 8 for a, b in zip(x0, x0[1:])) and (nseg - 1) * seg_h < ny <= nseg * seg_h
    assert x0[-2] + base + (quantum if ncol - 1 < extra else 0) - pad == nx
    col = [i for i in range(ncol) for _ in range(x0[i], x0[i + 1])]
    cols = [{col[x % nx] for x in range(x0[i] - 4, x0[i] - 4 + window) if -4 <= x < nx + 4} for i in range(ncol)]
    rows = [{(y % ny) // seg_h for y in range(g * seg_h - 4, min(ny, (g + 1) * seg_h) + 5)
             if 0 <= y < ny or (not walls and -4 <= y < ny + 4)} for g in range(nseg)]
    lists = [set(idx[ofs[t]:ofs[t + 1]]) for t in range(ncol * nseg)]
    bad = 0
    for g in range(nseg):
        for i in range(ncol):
            t = i + ncol * g
            for h in rows[g]:
                for c in cols[i]:
                    w = c + ncol * h
                    bad += (w not in lists[t]) + (t not in lists[w])
    return bad


def _lists(p):
    """nitems and the lists of a MultiArgs."""
    n = struct.unpack_from("<i", p, 0)[0]
    done, po, pi = struct.unpack_from("<3Q", p, 16)
    ofs = list((C.c_int32 * (n + 1)).from_address(po))
    return n, done, ofs, list((C.c_int32 * ofs[n]).from_address(pi))


def _single(fake, case):
    prec, tau, nx, ny, walls, sms, seg = CASES[case]
    fake.rt.fake_sms(sms)
    import paper_1307_6703_gb300 as lbm
    h = lbm.lb_create(lbm.lb_params(nx, ny, walls, prec, 0.375, 1 / 3, 0.3, 0.1, tau, 1e-4, 32.0, 0.0, 0.0, 0.3, 2.0, 0.0, None))
    lbm.lb_init(h, 0, 1, 1.0, 0.01)
    if seg:
        lbm.lb_set_seg_h(h, seg)
    out = {}

    def on_launch(name, grid, args):
        if "sweep_multi_kernel" in name:
            geo = _tiles(C.string_at(args[4], 56))
            n, done, ofs, idx = _lists(C.string_at(args[5], 64))
            boxes = {struct.unpack_from("<2I", C.string_at(args[k], 8)) for k in range(4)}
            out.update(tiles=n, expect=geo[4] * geo[5], boxes=sorted(boxes), room=fake.room(done) // 4,
                       missing=_missing(geo, 4 if prec == FP32 else 8, max(b[0] for b in boxes), ofs, idx))
    fake.on_launch = on_launch
    lbm.lb_step(h, 2)
    return out


@pytest.mark.parametrize("case", CASES)
def test_lists_cover_what_the_boxes_read(case, tmp_path):
    out = host_call(__file__, case, tmp_path)
    assert out["tiles"] == out["expect"] == out["room"]
    assert out["boxes"] == [[64, 2]]
    assert out["missing"] == 0


def _batch(fake, _):
    """The same for the work list of a batch: its items name lattice and tile."""
    import paper_1307_6703_gb300 as lbm
    dims = [(512, 256, 1), (64, 32, 0), (8, 8, 1), (1024, 64, 0)]
    b = lbm.Batch([lbm.lb_params(nx, ny, w, FP32, 0.375, 1 / 3, 0.3, 0.1, 1.0, 1e-4, 32.0, 0.0, 0.0, 0.3, 2.0, 0.0, None)
                   for nx, ny, w in dims])
    for v in b:
        v.init_noise(1, 1.0, 0.01)
    out = {"missing": 0, "tiles": 0, "expect": 0}

    def on_launch(name, grid, args):
        if "sweep_batch_multi" not in name:
            return
        items, sa = (C.cast(args[i], C.POINTER(C.c_void_p))[0] for i in (0, 1))
        n, done, ofs, idx = _lists(C.string_at(args[4], 64))
        it = [list((C.c_int32 * 5).from_address(items + 20 * j)) for j in range(n)]
        size = fake.room(sa) // (2 * len(dims))
        out["tiles"] = n
        for i in range(len(dims)):
            geo = _tiles(C.string_at(sa + 2 * i * size, 56))
            ncol = geo[5]
            tile = {j: v[1] + ncol * v[2] for j, v in enumerate(it) if v[0] == i}
            lists = [[] for _ in tile]
            for j, t in tile.items():
                lists[t] = [tile[d] for d in idx[ofs[j]:ofs[j + 1]]]   # (KeyError: another lattice's item)
            o = [0]
            for v in lists:
                o.append(o[-1] + len(v))
            out["expect"] += geo[4] * ncol
            out["missing"] += _missing(geo, 4, 64, o, sum(lists, []))
    fake.on_launch = on_launch
    b.step(2)
    return out


def test_lists_of_a_batch(tmp_path):
    out = host_call(__file__, "batch", tmp_path)
    assert out["tiles"] == out["expect"] > 0 and out["missing"] == 0


if __name__ == "__main__":
    os.makedirs(sys.argv[2], exist_ok=True)
    print(json.dumps((_batch if sys.argv[1] == "batch" else _single)(Fake(sys.argv[2]), sys.argv[1])))
