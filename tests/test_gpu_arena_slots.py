"""Arena slots that a record kernel reserves and leaves unused: the lane-group
forms (lane per component up to 9728 Lorenz / Van der Pol trajectories, 16 lanes
per neural Robertson trajectory) run more warps than a lane per trajectory does,
and must not need more of the arena for it. An ensemble that a lane per
trajectory fits into the fixed array of gs_solve_grad_noalloc still does, and a
record of at most the expected steps is made in one pass (its first arena)."""
import numpy as np
import pytest
import torch

from paper_2609_02876_gb300 import _native as N
from paper_2609_02876_gb300 import api, build
from paper_2609_02876_gb300 import workloads as W
from tests.test_gpu_tsit5 import dev
from tests.test_zz_no_alloc import _lib, _noalloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def steps(problem, P, Y, wl, t1, **kw):
    g = api.solve(problem, P, Y, wl["t0"], t1, [t1], wl["rtol"], wl["atol"], layout="soa", step_counts=True, **kw)
    return g["step_counts"][0].to(torch.int64)


def span_for(count, lo, hi, t_lo, t_hi):
    """A final time whose count lies in [lo, hi] (the count grows with the span)."""
    for _ in range(60):
        t = float(np.sqrt(t_lo * t_hi))
        c = count(t)
        if lo <= c <= hi:
            return t
        t_lo, t_hi = (t, t_hi) if c < lo else (t_lo, t)
    raise AssertionError("no span found")


@pytest.mark.parametrize("problem,d", [("lorenz", 3), ("vdp", 2)])
def test_noalloc_takes_what_a_lane_per_trajectory_fits(problem, d):
    n, mx, k = 9728, 16384, 14 - d
    wl = W.make(problem, n)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    # the array: counters, head, three words and eight doubles of y(t1) per trajectory, then 128-byte segments
    cap = ((32 << 20) - 256 - mx * (8 + 3 * 4 + 8 * 8)) // 128
    room = cap - 31 * ((n + 31) // 32)  # 31 slots unused in each of a lane per trajectory's warps
    t1 = span_for(lambda t: int(((steps(problem, P, Y, wl, t) + k - 1) // k).sum()), room - 600, room,
                  wl["t1"], 64 * wl["t1"])
    w = dict(wl, t1=t1, save_t=np.array([t1]))
    rc, out = _noalloc(_lib(), w, P, Y)
    assert rc == N.GS_OK, N.status_string(rc)
    rec, _, _ = api.forward_record(problem, P, Y, w["t0"], t1, [t1], w["rtol"], w["atol"], layout="soa",
                                   want_saves=False, ckpt_k=k)
    g = api.reverse(rec, P, Y, layout="soa")
    for key in ("loss", "params_bar", "y0_bar"):
        assert torch.equal(out[key], g[key]), key


@pytest.mark.parametrize("problem,n,expected", [("lorenz", 9728, 48 + 1), ("lorenz", 1024, 48 + 1), ("nrob", 128, 256)])
def test_records_of_the_expected_steps_keep_their_first_arena(problem, n, expected):
    wl = W.make(problem, n)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    kw = {}
    if problem == "nrob":
        kw["shared_w"] = torch.as_tensor(np.asarray(wl["w"], dtype=np.float32), device="cuda")
    t1 = span_for(lambda t: int(steps(problem, P, Y, wl, t, **kw).sum()), int(0.985 * expected * n), expected * n,
                  wl["t1"] / 8, 64 * wl["t1"])

    def record(t):
        # (a tolerance that no other record has: a freed one's arena may have grown)
        return api.forward_record(problem, P, Y, wl["t0"], t, [t], wl["rtol"] * (1 - 1e-9), wl["atol"], layout="soa",
                                  want_saves=False, ckpt_k=1, **kw)[0]

    short, full = record(t1 / 4), record(t1)
    assert full.bytes() == short.bytes()  # (a rerun's arena is sized to the demand)
