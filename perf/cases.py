"""The calls whose speed this framework is judged by: gradients (and solves) of
ODE ensembles through the package's public entry points.

A case is an entry point (`call`), a problem, an ensemble size `n`, a relative
tolerance, a precision and an array layout:

 - "solve_grad": record + reverse sweep with the built-in loss, the main call;
 - "autograd":   a training step through odeint_ensemble (forward, the user's
                 own loss on the saved states, backward);
 - "solve":      the forward-only solve (final states, nothing recorded);
 - "context":    solve_grad on a Context, what the request server runs for each
                 request.

The problems, parameter distributions, save times and tolerances are those of
workloads.py and bench.py. Inputs are drawn on the GPU from the seed.
"""
import math

import torch

from paper_2609_02876_gb300 import api

F64 = torch.float64

# problem: state dimension, parameters, time span, save times, absolute
# tolerance as a multiple of rtol (None: 1e-10), shared weights, accepted steps
# per trajectory at rtol 1e-6 (work estimates), order of the step count in rtol
PROBLEMS = {
    "lorenz": dict(d=3, P=3, t0=0.0, t1=1.0, ns=10, log=False, steps=45),
    "vdp": dict(d=2, P=1, t0=0.0, t1=10.0, ns=50, log=False, steps=95),
    "robertson": dict(d=3, P=3, t0=1e-5, t1=1e5, ns=20, log=True, steps=97),
    "hires": dict(d=8, P=12, t0=0.0, t1=321.8122, ns=10, log=False, steps=196),
    "lv_ude": dict(d=2, P=2, t0=0.0, t1=5.0, ns=10, log=False, steps=32),
    "nrob": dict(d=3, P=2, t0=1e-5, t1=1e5, ns=20, log=True, steps=243),
}
STIFF = ("robertson", "hires", "nrob")
HIRES_RATES = (1.71, 0.43, 8.32, 0.0007, 8.75, 10.03, 0.035, 1.12, 1.745, 280.0, 0.69, 1.81)


def _case(name, call, problem, n, rtol=1e-6, precision="fp64", layout="soa"):
    return dict(name=name, call=call, problem=problem, n=n, rtol=rtol, precision=precision, layout=layout)


def listed():
    return [
        # a parameter study of a thousand trajectories, interactive: latency counts
        _case("lorenz grad 1024", "solve_grad", "lorenz", 1024, layout="aos"),
        # one request of the serving stream, small and at the tight tolerance
        _case("vdp request 700", "context", "vdp", 700, rtol=1e-8),
        # fitting the neural Robertson at the paper's batch of 128 trajectories
        _case("nrob grad 128", "solve_grad", "nrob", 128, layout="aos"),
        # one gradient of a neural-ODE fit: shared network weights over a mid-size ensemble
        _case("lv_ude grad 2^16", "solve_grad", "lv_ude", 1 << 16, precision="fp32_mixed"),
        # a training step of the user's own loss on observations, odd batch
        _case("lorenz train 10007", "autograd", "lorenz", 10007, layout="aos"),
        # the non-stiff sweep's lower end, many saves, trajectories of very different length
        _case("vdp grad 65521", "solve_grad", "vdp", 65521),
        # stiff kinetics, the small and the large system
        _case("robertson grad 2^18", "solve_grad", "robertson", 1 << 18),
        _case("hires grad 30000", "solve_grad", "hires", 30000),
        # screening a million initial conditions: final states only
        _case("lorenz solve 10^6", "solve", "lorenz", 1000003),
        # the sweep's loose-tolerance corner in the mixed precision
        _case("vdp mixed 10^6", "solve_grad", "vdp", 1000000, rtol=1e-4, precision="fp32_mixed"),
        # the largest ensembles, in both precisions
        _case("lorenz mixed 2^24", "solve_grad", "lorenz", 1 << 24, precision="fp32_mixed"),
        _case("lorenz grad 2^24", "solve_grad", "lorenz", 1 << 24),
    ]


def _log_size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n | 1 if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(("small", "request", "nrob", "lv_ude", "train", "nonstiff", "robertson", "hires", "solve",
                       "mixed", "mixed"))
    rtol = rng.choice((1e-4, 1e-6, 1e-6, 1e-8))
    layout = rng.choice(("soa", "aos"))
    nonstiff = rng.choice(("lorenz", "vdp"))
    if kind == "small":
        c = _case("", "solve_grad", rng.choice(("lorenz", "vdp", "robertson")), _log_size(rng, 64, 1 << 14), rtol)
    elif kind == "request":
        c = _case("", "context", rng.choice(("lorenz", "vdp", "robertson")), _log_size(rng, 64, 1 << 16),
                  rng.choice((1e-6, 1e-8)))
    elif kind == "nrob":
        c = _case("", "solve_grad", "nrob", _log_size(rng, 32, 2048))
    elif kind == "lv_ude":
        c = _case("", "solve_grad", "lv_ude", _log_size(rng, 1 << 12, 1 << 18), precision="fp32_mixed")
    elif kind == "train":
        c = _case("", "autograd", nonstiff, _log_size(rng, 1 << 10, 1 << 17))
    elif kind == "nonstiff":
        c = _case("", "solve_grad", nonstiff, _log_size(rng, 1 << 14, 1 << 21), rtol)
    elif kind == "robertson":
        c = _case("", "solve_grad", "robertson", _log_size(rng, 1 << 12, 1 << 19), rng.choice((1e-6, 1e-8)))
    elif kind == "hires":
        c = _case("", "solve_grad", "hires", _log_size(rng, 1 << 12, 1 << 17))
    elif kind == "solve":
        c = _case("", "solve", nonstiff, _log_size(rng, 1 << 10, 1 << 21), rtol, rng.choice(("fp64", "fp32_mixed")))
    else:
        c = _case("", "solve_grad", nonstiff, _log_size(rng, 1 << 16, 1 << 23), rng.choice((1e-4, 1e-6)), "fp32_mixed")
    c["layout"] = layout
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _save_times(pr):
    t0, t1, ns = pr["t0"], pr["t1"], pr["ns"]
    if pr["log"]:
        a, b = math.log10(t0), math.log10(t1)
        s = [10.0 ** (a + (b - a) * j / ns) for j in range(1, ns + 1)]
    else:
        s = [t0 + (t1 - t0) * j / ns for j in range(1, ns + 1)]
    s[-1] = t1
    return s


def _atol(case):
    return 1e-10 if case["problem"] in STIFF else 1e-2 * case["rtol"]


def _ensemble(case, seed):
    """params [P][n], y0 [d][n] and the shared weights (or None), on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, problem = case["n"], case["problem"]

    def uni(lo, hi):
        return lo + (hi - lo) * torch.rand(n, dtype=F64, device="cuda", generator=g)

    def const(v):
        return torch.full((n,), v, dtype=F64, device="cuda")

    def glorot(fan_in, fan_out):
        a = math.sqrt(6.0 / (fan_in + fan_out))
        return a * (2.0 * torch.rand(fan_in * fan_out, dtype=F64, device="cuda", generator=g) - 1.0)

    def zeros(m):
        return torch.zeros(m, dtype=F64, device="cuda")

    w = None
    if problem == "lorenz":
        p = [uni(8, 12), uni(20, 30), uni(2, 3)]
        y = [1.0 + 0.1 * torch.randn(n, dtype=F64, device="cuda", generator=g) for _ in range(3)]
    elif problem == "vdp":
        p, y = [uni(0.5, 2)], [uni(-2, 2), uni(-2, 2)]
    elif problem == "robertson":
        p = [k * torch.exp(uni(math.log(0.9), math.log(1.1))) for k in (0.04, 3e7, 1e4)]
        y = [const(1.0), const(0.0), const(0.0)]
    elif problem == "hires":
        p = [k * torch.exp(uni(math.log(0.9), math.log(1.1))) for k in HIRES_RATES]
        y = [const(v) for v in (1.0, 0, 0, 0, 0, 0, 0, 0.0057)]
    elif problem == "lv_ude":
        p, y = [uni(1, 1.5), uni(2, 3)], [uni(0.5, 2), uni(0.5, 2)]
        w = torch.cat([glorot(2, 16), zeros(16), glorot(16, 16), zeros(16), glorot(16, 2), zeros(2)])
    else:
        p, y = [uni(0.04, 0.06), const(1e4)], [const(1.0), const(0.0), const(0.0)]
        w = torch.cat([glorot(3, 16), zeros(16), glorot(16, 16), zeros(16), glorot(16, 1), zeros(1) - 9.0])
    return torch.stack(p), torch.stack(y), None if w is None else w.to(torch.float32)


def _observations(case, seed, y0):
    """Observed states of a fit at the save times, (n, ns, d): the initial state with noise of the attractor's size."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    pr = PROBLEMS[case["problem"]]
    noise = torch.randn((case["n"], pr["ns"], pr["d"]), dtype=F64, device="cuda", generator=g)
    return y0.t()[:, None, :] + 2.0 * noise


def prepare(case, seed):
    pr = PROBLEMS[case["problem"]]
    p, y, w = _ensemble(case, seed)
    st = dict(case=case, w=w, save_t=_save_times(pr), t0=pr["t0"], t1=pr["t1"], rtol=case["rtol"], atol=_atol(case))
    if case["call"] == "autograd":
        st["obs"] = _observations(case, seed, y)
    if case["call"] == "context":
        st["ctx"] = api.Context()
    if case["layout"] == "aos" or case["call"] == "autograd":  # odeint_ensemble takes (n, P), (n, d)
        p, y = p.t().contiguous(), y.t().contiguous()
    st["params"], st["y0"] = p, y
    return st


def run(st):
    c = st["case"]
    head = (c["problem"], st["params"], st["y0"], st["t0"], st["t1"])
    tol = (st["rtol"], st["atol"])
    if c["call"] == "autograd":
        p, y = st["params"].detach().requires_grad_(), st["y0"].detach().requires_grad_()
        ys = api.odeint_ensemble(c["problem"], p, y, st["t0"], st["t1"], st["save_t"], *tol, precision=c["precision"])
        loss = (ys - st["obs"]).square().sum()
        loss.backward()
        return {"y_save": ys.detach(), "loss": loss.detach(), "params_bar": p.grad, "y0_bar": y.grad}
    kw = dict(layout=c["layout"], precision=c["precision"], shared_w=st["w"])
    if c["call"] == "solve":
        r = api.solve(*head, [], *tol, want_saves=False, **kw)
        return {"y_final": r["y_final"], "status": r["status"]}
    if c["call"] == "context":
        r = st["ctx"].solve_grad(*head, st["save_t"], *tol, **kw)
    else:
        r = api.solve_grad(*head, st["save_t"], *tol, **kw)
    return {k: r[k] for k in ("loss", "params_bar", "y0_bar", "shared_w_bar", "status") if k in r}


# ---------------------------------------------------------------------------
# Work: inputs read and outputs written once; the flops of the steps (an FMA
# counts two), with the right-hand side's f, its VJP, Jacobian and the
# contraction of its second derivatives counted by hand.
# ---------------------------------------------------------------------------
RHS_FLOPS = {"lorenz": (8, 20, 0, 0), "vdp": (5, 15, 0, 0), "robertson": (8, 21, 7, 24), "hires": (38, 88, 6, 78),
             "lv_ude": (804, 1554, 0, 0), "nrob": (854, 2400, 1700, 3800)}


def work(case):
    pr = PROBLEMS[case["problem"]]
    n, D, P, ns = case["n"], pr["d"], pr["P"], pr["ns"]
    f, vjp, jac, con = RHS_FLOPS[case["problem"]]
    steps = pr["steps"] * (1e-6 / case["rtol"]) ** 0.2
    if case["problem"] in STIFF:
        trial = jac + D + 2 * D ** 3 / 3 + 56 * D + 8 * f + 70 * D + 16 * D * D + D
        rev = 7 * D + 16 * D * D + 8 * D + 112 * D + 8 * vjp + 8 * D + 8 * con
    else:
        trial, rev = 7 * f + 68 * D + 4, 6 * vjp + 54 * D
    if case["call"] == "solve":
        return {"bytes": n * (8 * (P + 2 * D) + 4), "flops": n * steps * trial}
    nbytes = n * 8 * (2 * (P + D) + 1) + 4 * n
    if case["call"] == "autograd":
        nbytes += 2 * 8 * n * ns * D
    return {"bytes": nbytes, "flops": n * (steps + ns - 1) * (trial + rev)}


# ---------------------------------------------------------------------------
# The same results in plain torch, 64 bits: the adaptive solve of each
# trajectory, then the loss as a function of (params, y0, weights) on the
# accepted step sizes held fixed, differentiated by torch's autograd.
# Arrays are [D, m] here.
# ---------------------------------------------------------------------------
TS_A = (  # Tsitouras (2011), Table 1; row 7 is b (first same as last)
    (0.161,),
    (-0.008480655492356989, 0.335480655492357),
    (2.897153057105493, -6.359448489975075, 4.3622954328695815),
    (5.325864828439257, -11.748883564062828, 7.4955393428898365, -0.09249506636175525),
    (5.86145544294642, -12.92096931784711, 8.159367898576159, -0.071584973281401, -0.028269050394068383),
    (0.09646076681806523, 0.01, 0.4798896504144996, 1.379008574103742, -3.290069515436081, 2.324710524099774))
TS_BHAT = (0.09468075576583945, 0.009183565540343, 0.4877705284247616, 1.234297566930479, -2.707712349983525,
           1.866628418170587, 1.0 / 66.0)
RO_GAMMA = 0.21193756319429014  # Rodas5P (Steinebach 2023), transformed coefficients
RO_A6 = (-7.502846399306121, 2.561846144803919, -11.627539656261098, -0.18268767659942256, 0.030198172008377946)
RO_A = ((), (3.0,), (2.849394379747939, 0.45842242204463923), (-6.954028509809101, 2.489845061869568, -10.358996098473584),
        (2.8029986275628964, 0.5072464736228206, -0.3988312541770524, -0.04721187230404641), RO_A6, RO_A6 + (1.0,),
        RO_A6 + (1.0, 1.0))
RO_C = ((), (-14.155112264123755,), (-17.97296035885952, -2.859693295451294),
        (147.12150275711716, -1.41221402718213, 71.68940251302358),
        (165.43517024871676, -0.4592823456491126, 42.90938336958603, -5.961986721573306),
        (24.854864614690072, -3.0009227002832186, 47.4931110020768, 5.5814197821558125, -0.6610691825249471),
        (30.91273214028599, -3.1208243349937974, 77.79954646070892, 34.28646028294783, -19.097331116725623,
         -28.087943162872662),
        (37.80277123390563, -3.2571969029072276, 112.26918849496327, 66.9347231244047, -40.06618937091002,
         -54.66780262877968, -9.48861652309627))


def _mlp(w, x, n_in, n_out):
    a, b = 16 * n_in, 16 * n_in + 16
    h = torch.tanh(w[:a].view(16, n_in) @ x + w[a:b, None])
    h = torch.tanh(w[b:b + 256].view(16, 16) @ h + w[b + 256:b + 272, None])
    return w[b + 272:b + 272 + 16 * n_out].view(n_out, 16) @ h + w[b + 272 + 16 * n_out:, None]


def _rhs(problem, w):
    def f(y, p):
        if problem == "lorenz":
            o = (p[0] * (y[1] - y[0]), y[0] * (p[1] - y[2]) - y[1], y[0] * y[1] - p[2] * y[2])
        elif problem == "vdp":
            o = (y[1], p[0] * ((1 - y[0] * y[0]) * y[1] - y[0]))
        elif problem == "robertson":
            a, b, c = p[0] * y[0], p[2] * y[1] * y[2], p[1] * y[1] * y[1]
            o = (b - a, a - b - c, c)
        elif problem == "nrob":
            r = p[1] * y[1] * y[2] - p[0] * y[0]
            c = torch.nn.functional.softplus(_mlp(w, y, 3, 1)[0], threshold=1e9)
            o = (r, -r - c, c)
        elif problem == "lv_ude":
            nn = _mlp(w, y, 2, 2)
            o = (p[0] * y[0] - nn[0], -p[1] * y[1] + nn[1])
        else:
            u = p[9] * y[5] * y[7]
            o = (-p[0] * y[0] + p[1] * y[1] + p[2] * y[2] + p[3], p[0] * y[0] - p[4] * y[1],
                 -p[5] * y[2] + p[1] * y[3] + p[6] * y[4], p[2] * y[1] + p[0] * y[2] - p[7] * y[3],
                 -p[8] * y[4] + p[1] * (y[5] + y[6]),
                 -u + p[10] * y[3] + p[0] * y[4] - p[1] * y[5] + p[10] * y[6], u - p[11] * y[6], p[11] * y[6] - u)
        return torch.stack(o)

    return f


def _combine(coef, ks):
    return sum(c * k for c, k in zip(coef, ks))


def _tsit5(f, y, p, h):
    k = [f(y, p)]
    for row in TS_A:
        yi = y + h * _combine(row, k)
        k.append(f(yi, p))
    return yi, h * _combine([b - bh for b, bh in zip(TS_A[5] + (0.0,), TS_BHAT)], k)


def _rodas5p(f, y, p, h):
    D = y.shape[0]
    eye = torch.eye(D, dtype=F64, device=y.device)
    cols = [torch.func.jvp(lambda x: f(x, p), (y,), (eye[:, c:c + 1].expand_as(y).contiguous(),))[1] for c in range(D)]
    W = eye / (h * RO_GAMMA)[:, None, None] - torch.stack(cols, -1).permute(1, 0, 2)  # [m, D, D]
    lu, piv = torch.linalg.lu_factor(W)
    U = []
    for a, c in zip(RO_A, RO_C):
        yi = y + _combine(a, U) if U else y
        r = f(yi, p) + _combine(c, U) / h if U else f(yi, p)
        U.append(torch.linalg.lu_solve(lu, piv, r.t()[..., None])[..., 0].t())
    return yi + U[7], U[7]


def _first_step(f, y, p, t0, t1, rtol, atol):
    """Hairer, Norsett & Wanner I, Sec. II.4, order 5."""
    def rms(v):
        return ((v / sc) ** 2).mean(0).sqrt()

    sc, f0 = atol + rtol * y.abs(), f(y, p)
    d0, d1 = rms(y), rms(f0)
    h0 = torch.where((d0 < 1e-5) | (d1 < 1e-5), torch.full_like(d0, 1e-6), 0.01 * d0 / d1).clamp(max=t1 - t0)
    d2 = rms(f(y + h0 * f0, p) - f0) / h0
    dm = torch.maximum(d1, d2)
    h1 = torch.where(dm <= 1e-15, (h0 * 1e-3).clamp(min=1e-6), (0.01 / dm) ** (1 / 6))
    return torch.minimum(100 * h0, h1).clamp(max=t1 - t0)


@torch.no_grad()
def _mesh(step, f, y, p, t0, t1, rtol, atol):
    """Accepted steps H [S_max, m] (the first step repeated past a trajectory's end) and their number S [m]."""
    m = y.shape[1]
    t, h = torch.full((m,), t0, dtype=F64, device=y.device), _first_step(f, y, p, t0, t1, rtol, atol)
    S = torch.zeros(m, dtype=torch.long, device=y.device)
    rej = torch.zeros(m, dtype=torch.bool, device=y.device)
    H = torch.zeros((128, m), dtype=F64, device=y.device)
    live = torch.ones_like(rej)
    lanes = torch.arange(m, device=y.device)
    for it in range(100000):
        if it % 16 == 0 and not bool(live.any()):
            break
        last = t + h >= t1 - 1e-12 * max(1.0, abs(t1))
        hh = torch.where(last & live, t1 - t, h)
        hh = torch.where(live, hh, H[0])
        yn, e = step(f, y, p, hh)
        q = ((e / (atol + rtol * torch.maximum(y.abs(), yn.abs()))) ** 2).mean(0)
        acc = live & (q <= 1)
        if it >= H.shape[0]:
            H = torch.cat([H, torch.zeros_like(H)])
        H[S[acc], lanes[acc]] = hh[acc]
        S = S + acc
        t = torch.where(acc, torch.where(last, torch.full_like(t, t1), t + hh), t)
        y = torch.where(acc, yn, y)
        fac = torch.where(q.isfinite(), (0.9 * q.clamp(min=1e-300) ** -0.1).clamp(0.2, 10.0), torch.full_like(q, 0.2))
        fac = torch.where(acc & rej, fac.clamp(max=1.0), fac)
        live = live & ~(acc & last)
        h, rej = torch.where(live, hh * fac, h), ~acc
    Smax = int(S.max())
    H = H[:Smax]
    used = torch.arange(Smax, device=y.device)[:, None] < S
    return torch.where(used, H, H[:1]), S


def _replay(step, f, y, p, t0, t1, save_t, H, S):
    """States at the save times, [ns, D, m]: the mesh's steps, then one step from the mesh point before each save."""
    t = torch.full_like(H[0], t0)
    states, times = [y], [t]
    for i in range(H.shape[0]):
        yn = step(f, y, p, H[i])[0]
        y = torch.where(i < S, yn, y)
        t = torch.where(i < S, torch.where(i == S - 1, torch.full_like(t, t1), t + H[i]), t)
        states.append(y)
        times.append(t)
    states, times = torch.stack(states), torch.stack(times)
    out = []
    for s in save_t:
        i = torch.minimum((times <= s).sum(0) - 1, S)
        base = states.gather(0, i[None, None].expand(1, *states.shape[1:]))[0]
        hs = s - times.gather(0, i[None])[0]
        out.append(torch.where(hs > 0, step(f, base, p, torch.where(hs > 0, hs, H[0]))[0], base))
    return torch.stack(out)


def exact(case, seed):
    pr, problem, n = PROBLEMS[case["problem"]], case["problem"], case["n"]
    steps = pr["steps"] * (1e-6 / case["rtol"]) ** 0.2
    heavy = {"robertson": 12, "hires": 60, "nrob": 40, "lv_ude": 8}.get(problem, 1) * (0.3 if case["call"] == "solve" else 1)
    if n * steps * heavy > 1.2e8:  # more than some twenty seconds
        return None
    p, y, w = _ensemble(case, seed)
    w = None if w is None else w.double().requires_grad_()
    f, step = _rhs(problem, w), _rodas5p if problem in STIFF else _tsit5
    t0, t1, saves = pr["t0"], pr["t1"], _save_times(pr)
    obs = _observations(case, seed, y) if case["call"] == "autograd" else None
    got, block = [], 8192 if problem in ("hires", "nrob") else 32768
    for k in range(0, n, block):
        pk, yk = (x[:, k:k + block].contiguous() for x in (p, y))
        H, S = _mesh(step, f, yk, pk, t0, t1, case["rtol"], _atol(case))
        if case["call"] == "solve":
            with torch.no_grad():
                got.append({"y_final": _replay(step, f, yk, pk, t0, t1, [t1], H, S)[0]})
            continue
        pk.requires_grad_()
        yk.requires_grad_()
        ys = _replay(step, f, yk, pk, t0, t1, saves, H, S)
        if obs is None:
            loss = ys.square().sum((0, 1))
        else:
            ys = ys.permute(2, 0, 1)
            loss = (ys - obs[k:k + block]).square().sum((1, 2))
        loss.sum().backward()
        got.append({"loss": loss.detach(), "params_bar": pk.grad, "y0_bar": yk.grad, "y_save": ys.detach()})
        del ys, loss
    g = {k: torch.cat([x[k] for x in got], 0 if (k == "y_save") else -1) for k in got[0] if k != "y_save" or obs is not None}
    if case["layout"] == "aos" or case["call"] == "autograd":
        g = {k: v.t().contiguous() if k in ("params_bar", "y0_bar", "y_final") else v for k, v in g.items()}
    if obs is not None:
        g["loss"] = g["loss"].sum()
    elif case["call"] != "solve":
        g["status"] = None
        if w is not None:
            g["shared_w_bar"] = w.grad
    if case["call"] == "solve":
        g["status"] = None
    return g
