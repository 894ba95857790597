"""The HIRES factorisation that skips structural zeros, against the FP64 oracle
(dense LU with the same pivoting) where its row exchanges differ: rate constants
that reorder the pivots, zero rates (empty columns, zero multipliers) and both
Rosenbrock methods; and what it makes of a singular or non-finite system."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_02876_gb300 import api, build
from paper_2609_02876_gb300 import workloads as W
from tests.test_gpu_tsit5 import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method,om", [("rodas5p", oracle.METHOD_RODAS5P),
                                       ("rosenbrock23", oracle.METHOD_ROSENBROCK23)])
@pytest.mark.parametrize("n", [1, 70])
def test_hires_pivot_orders_match_the_oracle(method, om, n):
    build.build()
    rng = np.random.RandomState(11)
    wl = W.make("hires", n)
    p = wl["params"] * 10.0 ** rng.uniform(-2.5, 2.5, (n, 12))  # pivots change rows
    p[rng.uniform(size=p.shape) < 0.1] = 0.0
    y = wl["y0"] + rng.uniform(0.0, 1.0, (n, 8)) * (rng.uniform(size=(n, 8)) < 0.7)
    saves = np.linspace(0.0, 2.0, 5)[1:]
    P, Y = dev(p.T), dev(y.T)
    rec, ysv, st = api.forward_record("hires", P, Y, 0.0, 2.0, saves, 1e-4, 1e-8, layout="soa", method=method)
    assert (st.cpu().numpy() == 0).all()
    g = api.reverse(rec, P, Y, layout="soa")
    off, h = rec.export_mesh()
    o = oracle.replay_grad("hires", p, y, 0.0, 2.0, saves, off, h, method=om)
    # normwise per trajectory vector, as the HIRES parity tests
    for got, ref in ((ysv.permute(2, 0, 1), o["y_save"]), (g["params_bar"].T, o["params_bar"]),
                     (g["y0_bar"].T, o["y0_bar"])):
        got, ref = got.cpu().numpy().reshape(n, -1), ref.reshape(n, -1)
        assert (np.abs(got - ref).max(1) <= 1e-10 * np.abs(ref).max(1)).all()


def test_non_finite_states_fail_as_before():
    build.build()
    wl = W.make("hires", 3)
    y = wl["y0"].copy()
    y[1, 4] = np.inf
    y[2, 0] = 1e308
    r = api.solve("hires", dev(wl["params"].T), dev(y.T), wl["t0"], wl["t1"], wl["save_t"], wl["rtol"], wl["atol"],
                  layout="soa", check=False, want_saves=False)
    s = r["status"].cpu().numpy()
    assert s[0] == 0 and s[1] == 3
