"""What a call chooses by the device memory that is free, with most of it taken,
and what the pool of freed records keeps."""
import numpy as np
import pytest
import torch

from paper_2609_02876_gb300 import api, build
from paper_2609_02876_gb300 import workloads as W
from tests.test_gpu_queueing import args
from tests.test_gpu_tsit5 import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def outputs(P, Y):
    n = P.shape[1]
    return {"loss": torch.empty(n, dtype=torch.float64, device="cuda"), "params_bar": torch.empty_like(P),
            "y0_bar": torch.empty_like(Y), "status": torch.empty(n, dtype=torch.int32, device="cuda")}


def take_all_but(gb):
    """A tensor that leaves about `gb` GB of the device free (not touched)."""
    return torch.empty(torch.cuda.mem_get_info()[0] - (gb << 30), dtype=torch.uint8, device="cuda")


def test_interval_after_a_packed_solve_follows_the_free_memory():
    """A context that holds a packed FP32-mixed arena (32-byte segments) takes an
    FP64 call, whose segments are larger: the arena it holds does not decide."""
    n = 1 << 20
    wl = W.make("vdp", n)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    out = outputs(P, Y)
    ctx = api.Context()
    info = np.zeros(2, np.int32)
    torch.cuda.empty_cache()
    hogs = [take_all_but(16)]
    try:
        ctx.solve_grad("vdp", P, Y, *args(wl), layout="soa", out=out, precision="fp32_mixed", record_info=info)
        assert tuple(info) == (1, 0)
        hogs.append(take_all_but(1))
        # 3.4 GB held: every state of the FP64 record would take 5.1 GB, a state in 12 steps 1.3 GB
        ctx.solve_grad("vdp", P, Y, *args(wl), layout="soa", out=out, record_info=info)
        assert tuple(info) == (14 - 2, 0)
        assert (out["status"] == 0).all()
    finally:
        hogs.clear()
        ctx.close()
        torch.cuda.empty_cache()


def test_pool_counts_the_weight_partials():
    """A neural Robertson record of 111 MiB has 26 MiB of weight-gradient partials
    besides: together more than the pool keeps, so freeing it gives all back."""
    wl = W.make("nrob", 9101)
    w = torch.as_tensor(np.asarray(wl["w"], dtype=np.float32), device="cuda")
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    used = []
    for n in (9100, 9101):  # (the first also loads the kernels)
        Pn, Yn = P[:, :n].contiguous(), Y[:, :n].contiguous()
        free = torch.cuda.mem_get_info()[0]
        rec, _, _ = api.forward_record("nrob", Pn, Yn, *args(wl), layout="soa", shared_w=w, want_saves=False)
        assert (100 << 20) < rec.bytes() < (128 << 20)
        rec.free()
        used.append(free - torch.cuda.mem_get_info()[0])
    assert used[1] < (16 << 20), used
