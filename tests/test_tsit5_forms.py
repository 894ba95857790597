"""The integer FP64 multiplication of the Tsit5 kernels (SoftD): bit for bit the
IEEE product on the CPU (where the compiler's multiplication is the reference),
its range test, and on the GPU the same results from ensembles that take it and
ones that do not, with values in and out of its range; and the lane-per-component
form of small ensembles against the per-lane forms."""
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2609_02876_gb300 import api, build as B
from paper_2609_02876_gb300 import workloads as W
from tests.test_gpu_tsit5 import dev

SRC = r"""
#include <cstdio>
#include <cstring>
#include "gs_device.cuh"
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static double val(uint64_t sign, uint64_t e, uint64_t m) {
  uint64_t u = (sign << 63) | (e << 52) | (m & 0xfffffffffffffull);
  double d; memcpy(&d, &u, 8); return d;
}
static int check(double a, double b) {
  uint64_t x, y, w; memcpy(&x, &a, 8); memcpy(&y, &b, 8);
  volatile double r = a * b; double rr = r; memcpy(&w, &rr, 8);
  uint32_t h, l;
  gs::soft_mul_words((uint32_t)(x >> 32), (uint32_t)x, (uint32_t)(y >> 32), (uint32_t)y, h, l);
  return (((uint64_t)h << 32) | l) != w;
}
int main() {
  long bad = 0;
  const uint64_t ones = 0xfffffffffffffull;
  for (long i = 0; i < 4000000; ++i) {  // random, short (ties), all-ones and near-power mantissas
    uint64_t m[2];
    for (int q = 0; q < 2; ++q) {
      m[q] = rnd() & ones;
      const int k = (i / 5 + 3 * q) % 5;
      if (k == 1) m[q] &= ones << (rnd() % 53);
      if (k == 2) m[q] = ones - (rnd() % 4);
      if (k == 3) m[q] = rnd() % 4;
    }
    bad += check(val(rnd() & 1, 512 + rnd() % 1023, m[0]), val(rnd() & 1, 512 + rnd() % 1023, m[1]));
  }
  const uint64_t es[] = {512, 513, 1022, 1023, 1024, 1533, 1534}, ms[] = {0, 1, ones, ones - 1, ones >> 1, 1ull << 51};
  for (uint64_t ea : es) for (uint64_t eb : es) for (uint64_t ma : ms) for (uint64_t mb : ms)
    for (int q = 0; q < 4; ++q) bad += check(val(q & 1, ea, ma), val(q >> 1, eb, mb));
  for (uint64_t e = 0; e < 2048; ++e) for (uint64_t m : ms) for (int q = 0; q < 2; ++q) {
    double d = val(q, e, m); uint64_t u; memcpy(&u, &d, 8);
    bad += gs::soft_range((uint32_t)(u >> 32)) != (e >= 512 && e <= 1534);
  }
  printf("%ld\n", bad);
  return bad != 0;
}
"""


def test_integer_product_is_the_ieee_product(tmp_path):
    src = tmp_path / "soft.cu"
    src.write_text(SRC)
    exe = str(tmp_path / "soft")
    r = subprocess.run([B.nvcc()] + B.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I",
                                              os.path.join(B.ROOT, "include"), str(src), "-o", exe],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout


def _grad(problem, p, y, wl, **kw):
    return api.solve_grad(problem, dev(p.T), dev(y.T), wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"],
                          layout="soa", check=False, **kw)


@pytest.mark.gpu
@pytest.mark.parametrize("control", ["fast", "fp64"])
@pytest.mark.parametrize("extreme", [False, True])
@pytest.mark.parametrize("n", [9729, 19457])
def test_lorenz_same_bits_on_both_sides_of_the_lines(n, extreme, control):
    """19457 trajectories take the integer products, 9729 the hardware ones, and
    the first 700 alone a lane per component: same bits, with trajectories on the
    z axis (zero states and slopes), at the origin, of tiny and of huge states,
    and with zero parameters."""
    B.build()
    m = 700
    wl = W.make("lorenz", n)
    p, y = wl["params"].copy(), wl["y0"].copy()
    if extreme:
        y[3] = (0.0, 0.0, 1.0)
        y[64] = 0.0
        y[65] = (1.0, 0.0, 0.0)
        y[96:128] *= 1e-180
        y[130] = (1e160, 1.0, 1.0)
        p[200] = 0.0
        p[201, 1] = 0.0
        y[260] = (np.inf, 1.0, 1.0)
        y[261] = (5e-324, 1e-310, 1.0)
    a = _grad("lorenz", p, y, wl, control=control)
    b = _grad("lorenz", p[:m], y[:m], wl, control=control)
    assert torch.equal(a["status"][:m], b["status"])
    for k in ("loss", "params_bar", "y0_bar"):
        assert torch.equal(a[k][..., :m].contiguous().view(torch.int64), b[k].contiguous().view(torch.int64)), k
    P, Y = dev(p.T), dev(y.T)
    args = (wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"])
    kw = dict(layout="soa", check=False, control=control)
    r1, s1, _ = api.forward_record("lorenz", P, Y, *args, ckpt_k=1, **kw)
    r2, s2, _ = api.forward_record("lorenz", P[:, :m].contiguous(), Y[:, :m].contiguous(), *args, ckpt_k=1, **kw)
    ok = b["status"] == 0
    assert torch.equal(s1[:, :, :m][:, :, ok], s2[:, :, ok])
    g1, g2 = api.reverse(r1, P, Y, layout="soa"), api.reverse(r2, P[:, :m].contiguous(), Y[:, :m].contiguous(), layout="soa")
    assert torch.equal(g1["params_bar"][:, :m][:, ok], g2["params_bar"][:, ok])  # the compact record's sweep
    f1 = api.solve("lorenz", P, Y, *args, **kw)
    f2 = api.solve("lorenz", P[:, :m].contiguous(), Y[:, :m].contiguous(), *args, **kw)
    assert torch.equal(f1["y_final"][:, :m][:, ok], f2["y_final"][:, ok])


@pytest.mark.gpu
@pytest.mark.parametrize("problem", ["lorenz", "vdp"])
@pytest.mark.parametrize("m", [1, 9, 31, 9728])
def test_lane_per_component_ragged_sizes(problem, m):
    """Up to 9728 trajectories run a lane per component, 9729 a lane each: same
    bits for ragged last groups and warps, user cotangents included."""
    B.build()
    wl = W.make(problem, 9729)
    P, Y = dev(wl["params"].T), dev(wl["y0"].T)
    args = (wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"])
    Ps, Ys = P[:, :m].contiguous(), Y[:, :m].contiguous()
    a = api.solve_grad(problem, P, Y, *args, layout="soa")
    b = api.solve_grad(problem, Ps, Ys, *args, layout="soa")
    for k in ("loss", "params_bar", "y0_bar"):
        assert torch.equal(a[k][..., :m], b[k]), k
    cot = torch.randn((len(wl["save_t"]), Y.shape[0], 9729), dtype=torch.float64, device="cuda",
                      generator=torch.Generator("cuda").manual_seed(1))
    for stages in (False, True):
        ra, ya, _ = api.forward_record(problem, P, Y, *args, layout="soa", record_stages=stages, ckpt_k=1)
        rb, yb, _ = api.forward_record(problem, Ps, Ys, *args, layout="soa", record_stages=stages, ckpt_k=1)
        assert torch.equal(ya[..., :m], yb)
        ga = api.reverse(ra, P, Y, cot, layout="soa")
        gb = api.reverse(rb, Ps, Ys, cot[..., :m].contiguous(), layout="soa")
        for k in ("params_bar", "y0_bar"):
            assert torch.equal(ga[k][:, :m], gb[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("problem,n", [("vdp", 1), ("vdp", 33), ("linear", 65)])
def test_two_dimensional_problems_with_zero_parameters_match_the_oracle(problem, n):
    """mu = 0 and triangular matrices: every unit leaves the integer range."""
    import oracle

    B.build()
    rng = np.random.RandomState(3)
    if problem == "vdp":
        p, t1 = np.where(np.arange(n)[:, None] % 2, rng.uniform(0.5, 2, (n, 1)), 0.0), 10.0
    else:
        p, t1 = rng.uniform(-1, 1, (n, 4)) * (np.arange(4) != 1), 2.0
    y = rng.uniform(0.5, 2, (n, 2))
    saves = np.linspace(0, t1, 6)[1:]
    P, Y = dev(p.T), dev(y.T)
    rec, _, st = api.forward_record(problem, P, Y, 0.0, t1, saves, 1e-6, 1e-8, layout="soa")
    assert (st.cpu().numpy() == 0).all()
    g = api.reverse(rec, P, Y, layout="soa")
    off, h = rec.export_mesh()
    o = oracle.replay_grad(problem, p, y, 0.0, t1, saves, off, h)
    for got, ref in ((g["params_bar"], o["params_bar"]), (g["y0_bar"], o["y0_bar"])):
        got = got.cpu().numpy().T
        assert (np.abs(got - ref).max(1) <= 1e-11 * np.abs(ref).max(1)).all()
