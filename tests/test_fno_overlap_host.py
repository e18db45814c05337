"""On which stream the weight gradients of the fused backward pass run (host
logic, on a CUDA runtime without a GPU): beside the rest for few fields, in turn
for many, and joined to the handle's stream either way."""
import json
import os
import sys

import pytest

from fake_cuda import STREAM, Fake, host_call


def _backward(fake, batch):
    from paper_1307_6703_gb300 import fno
    net = fno.Fno(layers=3, modes_x=8, modes_y=4, batch_max=batch, nx_max=16, ny_max=16, stream=STREAM)
    dev = fake.device(batch * 16 + 4 * batch * 3 * 256)
    fno.fno_forward(net.h, batch, 16, 16, dev, dev + batch * 16)
    fake.clear()
    net.backward(dev + batch * 16, want_loss=False)
    calls = [c for c in fake.calls if c[3] or c[0].startswith(("cudaEvent", "cudaStreamWait"))]
    last = max((i for i, c in enumerate(calls) if c[1] != STREAM), default=-1)
    joined = [c[0] for c in calls[last:] if c[0] == "cudaStreamWaitEvent" and c[1] == STREAM]
    return {"beside": sum("gemm_tn" in c[0] and c[1] != STREAM for c in calls), "joined": len(joined) > 0,
            "waits": sum(c[0] == "cudaStreamWaitEvent" for c in calls)}


@pytest.mark.parametrize("batch", [1, 24, 25, 64])
def test_weight_gradients_beside_or_in_turn(batch, tmp_path):
    out = host_call(__file__, str(batch), tmp_path)
    if batch <= 24:
        assert out["beside"] == 4 and out["joined"]      # dW of three layers and of the projection
    else:
        assert out["beside"] == 0 and out["waits"] == 0


if __name__ == "__main__":
    os.makedirs(sys.argv[2], exist_ok=True)
    print(json.dumps(_backward(Fake(sys.argv[2]), int(sys.argv[1]))))
