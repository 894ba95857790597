"""The solve call that queues the reverse sweep behind the record, and the pool
of freed records: an arena that turns out too small reruns both, outputs that
overlap the inputs, and records that reuse a freed one's buffers."""
import numpy as np
import pytest
import torch

from paper_2609_02876_gb300 import api, build
from paper_2609_02876_gb300 import workloads as W
from tests.test_gpu_tsit5 import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def long_lorenz(n, t1=9.0):
    """Nine times the usual span: several times the expected steps, so the first arena overflows."""
    wl = W.make("lorenz", n)
    return dict(wl, t1=t1, save_t=np.linspace(0.0, t1, 11)[1:])


def args(wl):
    return wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"]


@pytest.mark.parametrize("n", [1, 700, 20011])
@pytest.mark.parametrize("in_place", [False, True])
def test_overflowing_arena_reruns_record_and_sweep(n, in_place):
    wl = long_lorenz(n)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    rec, _, _ = api.forward_record("lorenz", P, Y, *args(wl), layout="soa", want_saves=False, ckpt_k=1)
    ref = api.reverse(rec, P, Y, layout="soa")
    p, y = P.clone(), Y.clone()
    out = {"loss": torch.empty(n, dtype=torch.float64, device="cuda"),
           "params_bar": p if in_place else torch.empty_like(P), "y0_bar": y if in_place else torch.empty_like(Y),
           "status": torch.full((n,), -1, dtype=torch.int32, device="cuda")}
    ctx = api.Context()  # a workspace of its own, so its first arena is the expected size
    g = ctx.solve_grad("lorenz", p, y, *args(wl), layout="soa", out=out)
    assert (g["status"] == 0).all()
    for k in ("loss", "params_bar", "y0_bar"):
        assert torch.equal(g[k], ref[k]), k
    ctx.close()


def test_failed_trajectories_keep_their_status_and_nan_gradients():
    wl = W.make("lorenz", 300)
    y = wl["y0"].copy()
    y[7] = np.nan
    g = api.solve_grad("lorenz", dev(wl["params"].T), dev(y.T), *args(wl), layout="soa", check=False)
    bad = g["status"] != 0
    assert bad.nonzero().flatten().tolist() == [7]
    assert torch.isnan(g["loss"][7]) and torch.isfinite(g["loss"][~bad]).all()


def test_records_from_the_pool_equal_fresh_ones():
    wl = W.make("lorenz", 3001)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    kw = dict(layout="soa", record_stages=True)
    r0, y0, _ = api.forward_record("lorenz", P, Y, *args(wl), **kw)
    g0, b0, s0 = api.reverse(r0, P, Y, layout="soa"), r0.bytes(), r0.stats()
    r1, y1, _ = api.forward_record("lorenz", P, Y, *args(wl), **kw)  # both alive: buffers of their own
    r0.free()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for i in range(6):
        q = P * (1.0 + 1e-3 * i)
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[i % 2]):
            r2, y2, _ = api.forward_record("lorenz", q, Y, *args(wl), **kw)
            g2 = api.reverse(r2, q, Y, layout="soa")
            assert r2.bytes() == b0
            r2.free()  # with the sweep still queued
        torch.cuda.synchronize()
        if i == 0:
            assert torch.equal(y2, y0) and all(torch.equal(g2[k], g0[k]) for k in ("loss", "params_bar", "y0_bar"))
    assert torch.equal(y1, y0) and r1.stats() == s0
    g1 = api.reverse(r1, P, Y, layout="soa")
    assert all(torch.equal(g1[k], g0[k]) for k in ("loss", "params_bar", "y0_bar"))
    # forward mode and a smaller ensemble after it, through the pool again
    fg = api.forward_grad(r1, P, Y, layout="soa")["params_bar"]
    r1.free()
    r3, _, _ = api.forward_record("lorenz", P, Y, *args(wl), **kw)
    assert torch.equal(api.forward_grad(r3, P, Y, layout="soa")["params_bar"], fg)
    r4, _, _ = api.forward_record("lorenz", P[:, :33].contiguous(), Y[:, :33].contiguous(), *args(wl), **kw)
    assert torch.equal(api.reverse(r4, P[:, :33].contiguous(), Y[:, :33].contiguous(), layout="soa")["params_bar"],
                       g0["params_bar"][:, :33])


def test_freeing_a_record_leaves_a_capture_alone():
    """A record may be freed (by the collector, say) while a stream captures in
    the relaxed mode; a sweep may be captured, and its record freed after the graph."""
    wl = W.make("lorenz", 2003)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    rec, _, _ = api.forward_record("lorenz", P, Y, *args(wl), layout="soa")
    ref = api.reverse(rec, P, Y, layout="soa")
    swept, _, _ = api.forward_record("lorenz", P, Y, *args(wl), layout="soa")
    torch.cuda.synchronize()
    graph, x = torch.cuda.CUDAGraph(), torch.zeros(4, device="cuda")
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        x.add_(1)
        rec.free()
        g = api.reverse(swept, P, Y, layout="soa")
        x.add_(1)
    other, _, _ = api.forward_record("lorenz", 1.01 * P, Y, *args(wl), layout="soa")  # through the pool
    graph.replay()
    torch.cuda.synchronize()
    assert (x == 2).all()
    for k in ("loss", "params_bar", "y0_bar"):
        assert torch.equal(g[k], ref[k]), k
    del graph
    swept.free()
    other.free()


@pytest.mark.parametrize("streams", [1, 3, 11])
def test_a_record_from_the_pool_waits_for_its_sweeps(streams):
    """A record freed with long sweeps queued on several streams, and its buffers
    taken by a record of other inputs on another stream: the sweeps' results stand."""
    wl = W.make("lorenz", 4001)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    kw = dict(layout="soa", record_stages=True)
    rec, _, _ = api.forward_record("lorenz", P, Y, *args(wl), **kw)
    ref = api.reverse(rec, P, Y, layout="soa")
    torch.cuda.synchronize()
    ss = [torch.cuda.Stream() for _ in range(streams)]
    out = []
    for s in ss:  # one stream's sweeps after the other's (a sweep's tickets are the record's own)
        s.wait_stream(torch.cuda.current_stream() if not out else prev)
        with torch.cuda.stream(s):
            out += [api.reverse(rec, P, Y, layout="soa") for _ in range(24 // streams)]
        prev = s
    rec.free()
    taker = torch.cuda.Stream()
    with torch.cuda.stream(taker):
        r2, _, _ = api.forward_record("lorenz", 1.5 * P, 0.5 * Y, *args(wl), **kw)
    torch.cuda.synchronize()
    for g in out:
        for k in ("loss", "params_bar", "y0_bar"):
            assert torch.equal(g[k], ref[k]), k
    r2.free()
