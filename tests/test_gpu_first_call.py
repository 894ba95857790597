"""A process's first call gives what its later calls give (each case runs in a
process of its own)."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2609_02876_gb300 import build

pytestmark = pytest.mark.gpu

NROB = r"""
import sys
import numpy as np, torch
from paper_2609_02876_gb300 import api, workloads as W
method, n, m = sys.argv[1], 30000, 15000
wl = W.make("nrob", n)
P, Y = (torch.as_tensor(np.ascontiguousarray(wl[k].T), device="cuda") for k in ("params", "y0"))
w = torch.as_tensor(np.asarray(wl["w"], dtype=np.float32), device="cuda")
def grad(lo, hi):
    return api.solve_grad("nrob", P[:, lo:hi].contiguous(), Y[:, lo:hi].contiguous(), wl["t0"], wl["t1"], wl["save_t"],
                          wl["rtol"], wl["atol"], layout="soa", shared_w=w, method=method)["shared_w_bar"].double()
first, again, a, b = grad(0, n), grad(0, n), grad(0, m), grad(m, n)
assert torch.equal(first, again), ((first - again).abs().max() / again.abs().max()).item()
# FP64 sums written out in FP32: half an ulp each
bound = 2.0 ** -23 * max(x.abs().max().item() for x in (first, a, b))
assert ((a + b) - first).abs().max().item() <= bound
"""


@pytest.mark.parametrize("method", ["rodas5p", "rosenbrock23"])
def test_first_weight_gradient_of_more_than_a_cta_per_sm(method):
    """The shared-weight gradient sums a partial of every warp that ran: 30000
    trajectories are more than one CTA per SM."""
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    r = subprocess.run([sys.executable, "-c", NROB, method], capture_output=True, text=True, timeout=600,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stderr[-2000:]
