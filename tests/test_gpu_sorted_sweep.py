"""gs_solve_grad sorts its reverse sweep by step count from one warp per FP64 unit on
(19456 trajectories on 152 SMs); a record handle's sweep takes the trajectories as they
come. Both do the same arithmetic per trajectory, so their gradients are equal bit for
bit, at the edges of the rule, for step counts past the sort's 1023 bins and with failed
trajectories."""
import numpy as np
import pytest
import torch

from paper_2609_02876_gb300 import api, build
from paper_2609_02876_gb300 import workloads as W
from tests.test_gpu_tsit5 import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("problem,n,span,fail", [
    ("vdp", 19456, 1, False), ("vdp", 19457, 1, True), ("lorenz", 38913, 1, False), ("robertson", 20011, 1, True),
    ("hires", 38912, 1, False), ("hires", 38913, 1, True), ("lorenz", 20011, 30, False)])
def test_same_as_unsorted(problem, n, span, fail):
    build.build()
    wl = W.make(problem, n)
    P, y0 = dev(wl["params"].T), np.array(wl["y0"].T)
    if fail:
        y0[0, 5::97] = np.nan
    Y = dev(y0)
    t1 = wl["t0"] + span * (wl["t1"] - wl["t0"])
    args = (wl["t0"], t1, wl["save_t"], wl["rtol"], wl["atol"])
    kw = dict(method=wl["method"]) if "method" in wl else {}
    rec, _, fwd = api.forward_record(problem, P, Y, *args, layout="soa", want_saves=False, ckpt_k=1, check=False, **kw)
    r = api.reverse(rec, P, Y, layout="soa")
    g = api.solve_grad(problem, P, Y, *args, layout="soa", check=False, step_counts=True, **kw)
    assert bool((g["status"] != 0).any()) == fail
    assert (int(g["step_counts"][0].max()) > 1023) == (span > 1)
    for k in ("loss", "params_bar", "y0_bar"):
        a, b = g[k].nan_to_num(7.0), r[k].nan_to_num(7.0)
        assert torch.equal(a, b), k


@pytest.mark.parametrize("problem,method,n", [("robertson", "rosenbrock23", 58369), ("nrob", None, 58368),
                                              ("nrob", None, 58369)])
def test_records_at_the_edge_of_three_waves(problem, method, n):
    """Where the record changes its CTAs per SM (58368 = 3 x 152 x 128 lanes): the last
    trajectories have the bits that they have among a few."""
    build.build()
    wl = W.make(problem, n)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    kw = dict(layout="soa", method=method)
    if wl["w"] is not None:
        kw["shared_w"] = torch.as_tensor(np.asarray(wl["w"], np.float32), device="cuda")

    def final(lo):
        p, y = P[:, lo:].contiguous(), Y[:, lo:].contiguous()
        args = (problem, p, y, wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"])
        if method:
            return api.solve_grad(*args, **kw)["params_bar"]
        return api.solve(*args, want_saves=False, **kw)["y_final"]

    assert torch.equal(final(0)[:, n - 30000:], final(n - 30000))
