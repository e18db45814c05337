"""Launch shapes of the network (host logic, on a CUDA runtime without a GPU): a
grid's y and z end at 65,535, whatever the fields' sizes."""
import json
import os
import sys

import pytest

from fake_cuda import Fake, host_call

# width, hidden, modes_x, fields, nx, ny
CASES = {
    "fused_tall": (32, 64, 8, 1, 16, 70000),
    "fused_tall_h32": (32, 32, 8, 2, 16, 65536),
    "fused_at_the_limit": (32, 64, 8, 1, 16, 65535),
    "fused_wide": (32, 64, 16, 1, 70008, 16),
    "fused_many": (32, 64, 8, 80, 16, 16),
    "separate_tall": (16, 64, 8, 1, 16, 70000),
}


def _grids(case, workdir):
    width, hidden, mx, batch, nx, ny = CASES[case]
    fake = Fake(workdir)
    from paper_1307_6703_gb300 import fno
    net = fno.Fno(width=width, hidden=hidden, layers=2, modes_x=mx, modes_y=4, outputs=3, batch_max=batch, nx_max=nx, ny_max=ny)
    dev = fake.device(batch * 16 + 4 * batch * 3 * nx * ny)
    fno.fno_forward(net.h, batch, nx, ny, dev, dev + batch * 16)
    net.backward(dev + batch * 16, want_loss=False)
    return [[name, *grid] for name, _, _, grid in fake.launches()]


@pytest.mark.parametrize("case", CASES)
def test_grids_are_within_the_limits(case, tmp_path):
    grids = host_call(__file__, case, tmp_path)
    names = " ".join(g[0] for g in grids)
    assert ("layer_kernel" in names) == case.startswith("fused")
    for name, x, y, z in grids:
        assert 1 <= x < 2 ** 31 and 1 <= y <= 65535 and 1 <= z <= 65535, (name, x, y, z)


if __name__ == "__main__":
    os.makedirs(sys.argv[2], exist_ok=True)
    print(json.dumps(_grids(sys.argv[1], sys.argv[2])))
