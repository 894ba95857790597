"""FP32-mixed solves over packed segments: the same bits as the general record
and sweep kernels (a record handle's), over sizes at the edges of warps and
blocks, both step controls, spans and save grids of every kind, and trajectories
that fail."""
import numpy as np
import pytest
import torch

from paper_2609_02876_gb300 import api, build
from paper_2609_02876_gb300 import workloads as W
from tests.test_gpu_queueing import args, long_lorenz
from tests.test_gpu_tsit5 import dev

pytestmark = pytest.mark.gpu


def both(problem, p, y, t0, t1, saves, rtol, atol, **kw):
    build.build()
    P, Y = dev(p.T), dev(y.T)
    kw = dict(layout="soa", precision="fp32_mixed", check=False, **kw)
    s = api.solve_grad(problem, P, Y, t0, t1, saves, rtol, atol, step_counts=True, **kw)
    rec, _, st = api.forward_record(problem, P, Y, t0, t1, saves, rtol, atol, ckpt_k=1, want_saves=False,
                                    step_counts=True, **kw)
    g = api.reverse(rec, P, Y, layout="soa")
    assert torch.equal(s["status"], st)
    assert torch.equal(s["step_counts"], rec.step_counts)
    for k in ("loss", "params_bar", "y0_bar"):
        assert torch.equal(s[k].view(torch.int64), g[k].view(torch.int64)), k
    return st.cpu().numpy()


@pytest.mark.parametrize("control", ["fast", "fp64"])
@pytest.mark.parametrize("problem", ["lorenz", "vdp"])
@pytest.mark.parametrize("n", [1, 31, 129, 40001])
def test_same_bits_as_the_general_kernels(problem, n, control):
    wl = W.make(problem, n)
    st = both(problem, wl["params"], wl["y0"], wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"],
              control=control)
    assert (st == 0).all()


@pytest.mark.parametrize("t0,t1,saves", [(0.0, 1.0, []), (-3.0, -1.0, [-2.5, -1.7]), (-1.0, 1.0, [-0.5, 1e-300, 1.0]),
                                         (2.0, 2.5, np.linspace(2.0, 2.5, 257)[1:])])
def test_spans_and_save_grids(t0, t1, saves):
    rng = np.random.RandomState(2)
    n = 333
    both("linear", rng.uniform(-1, 1, (n, 4)), rng.uniform(-1, 1, (n, 2)), t0, t1, saves, 1e-5, 1e-7)
    wl = W.make("lorenz", n)
    both("lorenz", wl["params"], wl["y0"], t0, t1, saves, 1e-5, 1e-7)


@pytest.mark.parametrize("n,rtol", [(3000001, 1e-6), (1 << 22, 1e-8)])
def test_large_ensembles_in_one_piece(n, rtol):
    """Up to the largest one-piece call and some 1e9 segments: parts solved alone have the same bits."""
    build.build()
    wl = W.make("vdp", n, rtol=rtol)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)

    def grad(lo, hi):
        return api.solve_grad("vdp", P[:, lo:hi].contiguous(), Y[:, lo:hi].contiguous(), wl["t0"], wl["t1"],
                              wl["save_t"], wl["rtol"], wl["atol"], layout="soa", precision="fp32_mixed")

    g = grad(0, n)
    for lo in (0, n // 2, n - 3000):
        part = grad(lo, lo + 3000)
        for k in ("loss", "params_bar", "y0_bar", "status"):
            assert torch.equal(g[k][..., lo:lo + 3000], part[k]), k


@pytest.mark.parametrize("kw", [dict(max_steps=20), dict(h0=1e-3), dict(h0=10.0)])
def test_options_and_failed_trajectories(kw):
    n = 777
    wl = W.make("lorenz", n)
    y = wl["y0"].copy()
    y[3] = np.nan
    y[64:96] = np.inf
    y[100] *= 1e30  # overflows single precision on the way
    y[101] = 0.0
    y[102] = 1e-37
    p = wl["params"].copy()
    p[200] = 0.0
    st = both("lorenz", p, y, wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"], **kw)
    assert (st[[3, 64, 95]] == 3).all()


@pytest.mark.parametrize("n", [1, 700, 20011])
@pytest.mark.parametrize("in_place", [False, True])
def test_overflowing_packed_arena_reruns_record_and_sweep(n, in_place):
    wl = long_lorenz(n)
    build.build()
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    rec, _, _ = api.forward_record("lorenz", P, Y, *args(wl), layout="soa", want_saves=False, ckpt_k=1,
                                   precision="fp32_mixed")
    ref = api.reverse(rec, P, Y, layout="soa")
    p, y = P.clone(), Y.clone()
    out = {"loss": torch.empty(n, dtype=torch.float64, device="cuda"),
           "params_bar": p if in_place else torch.empty_like(P), "y0_bar": y if in_place else torch.empty_like(Y),
           "status": torch.empty(n, dtype=torch.int32, device="cuda")}
    ctx = api.Context()  # a workspace of its own, so its first arena is the expected size
    g = ctx.solve_grad("lorenz", p, y, *args(wl), layout="soa", out=out, precision="fp32_mixed")
    assert (g["status"] == 0).all()
    for k in ("loss", "params_bar", "y0_bar"):
        assert torch.equal(g[k], ref[k]), k
    ctx.close()


def test_more_segments_than_a_packed_index_holds():
    """2.0e9 accepted steps where 2.1e8 were expected: past a packed segment's
    31-bit index, so the rerun is over general segments (about 110 GB)."""
    build.build()
    n = 1 << 21
    wl = W.make("vdp", n)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)

    def grad(ctx, lo, hi, t1, **kw):
        saves = np.linspace(0.0, t1, 6)[1:]
        return ctx.solve_grad("vdp", P[:, lo:hi].contiguous(), Y[:, lo:hi].contiguous(), 0.0, t1, saves, wl["rtol"],
                              wl["atol"], layout="soa", precision="fp32_mixed", **kw)

    ctx = api.Context()
    m = 1 << 17  # a packed sample gives the steps per unit of time
    s = grad(ctx, 0, m, 100.0, step_counts=True)["step_counts"][0].double().mean().item()
    t1 = 100.0 * 2.0e9 / (s * n)
    part = grad(ctx, n - m, n, t1, step_counts=True)
    total = part["step_counts"][0].double().mean().item() * n
    assert 1.93e9 < total < 2.1e9
    ctx.close()
    torch.cuda.empty_cache()
    ctx = api.Context()
    g = grad(ctx, 0, n, t1)
    assert (g["status"] == 0).all()
    for k in ("loss", "params_bar", "y0_bar", "status"):
        assert torch.equal(g[k][..., n - m:], part[k]), k
    used = torch.cuda.mem_get_info()[0]
    ctx.close()
    assert torch.cuda.mem_get_info()[0] - used > (90 << 30)  # the arena was the general one
