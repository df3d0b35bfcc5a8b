"""Performance cases: the calls that a program fitting Gaussian processes to
integrated, possibly overlapping exposures makes, through the package's public
entry points.

A case is a dict of plain values:

  call       entry point: "loglik", "grad" (Model.loglik_grad), "graph" (the
             same replayed from a CUDA graph), "host" (host buffers, the event
             stream sent again), "fit" (the autograd function and its backward
             pass), "windows" (with the gradient of the exposure windows),
             "condition", "predict"
  terms      kernel: "sho", "sho+m32", "sho+sho", "prod" or "prod+m32"
  slots      0: instantaneous measurements; k: exposures of k instruments,
             which overlap one another for k > 1
  layout     integral states: 0 one per slot, 1 one per term
  series     number of series, of n_min..n_max measurements each (log-uniform)
  sets       0: one hyperparameter vector per series; k: k vectors, each
             applied to every series
  low_q      quality factors around 0.6, so that some oscillators are overdamped
  precision  32 or 64
  stars      "predict": test times per series

Exposure recipes, kernels and sizes are those of ``synth`` and bench.py.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2601_02527_gb300 as gp

TWO_PI = 2.0 * math.pi
TERMS = {"sho": (gp.SHO,), "sho+m32": (gp.SHO, gp.MATERN32), "sho+sho": (gp.SHO, gp.SHO),
         "prod": (gp.SHO_PRODUCT,), "prod+m32": (gp.SHO_PRODUCT, gp.MATERN32)}

# centres of the hyperparameters; the white-noise sd follows them
_SHO = (1.0, TWO_PI / 10, 3.0)
_SHO2 = (0.5, TWO_PI / 2, 1.0)
_M32 = (0.5, 5.0)
_PROD = (1.0, TWO_PI / 50, 1.0, TWO_PI / 5, 10.0)
CENTRE = {"sho": _SHO, "sho+m32": _SHO + _M32, "sho+sho": _SHO + _SHO2,
          "prod": _PROD, "prod+m32": _PROD + _M32}
QUALITY = {"sho": (2,), "sho+m32": (2,), "sho+sho": (2, 5), "prod": (2, 4), "prod+m32": (2, 4)}
WHITE = 0.1


def _case(name, call, terms, slots, series, n_min, n_max, sets=0, layout=0, low_q=False,
          precision=32, stars=0):
    case = {"call": call, "terms": terms, "slots": slots, "layout": layout, "series": series,
            "n_min": n_min, "n_max": n_max, "sets": sets, "low_q": low_q,
            "precision": precision, "stars": stars}
    return {"name": name, **case} if name else case


def listed():
    return [
        # one star, one evaluation: the likelihood inside a sampler or a line search
        _case("single_loglik", "loglik", "sho", 1, 1, 1000, 1000),
        # a few short series, with the gradient of their exposure windows
        _case("windows", "windows", "sho+sho", 1, 8, 300, 1100, layout=1),
        # a survey's light curves, likelihood only
        _case("batch_loglik", "loglik", "sho+m32", 1, 1024, 500, 20000),
        # a survey with gradients: bench.py's headline workload
        _case("batch_grad", "grad", "sho+sho", 1, 1024, 2000, 20000, layout=1),
        # new data every step, from host memory
        _case("host_grad", "host", "sho+m32", 1, 255, 1000, 9001),
        # one long series of three overlapping instruments
        _case("long_loglik", "loglik", "sho", 3, 1, 1 << 20, 1 << 20),
        # walkers of an ensemble on one series of three instruments, from a graph
        _case("walkers_graph", "graph", "sho+m32", 3, 1, 50001, 50001, sets=48),
        # instantaneous measurements, one optimiser step by autograd
        _case("instants_fit", "fit", "sho+m32", 0, 700, 500, 15000),
        # conditioned mean and variance of every measurement of two instruments
        _case("condition", "condition", "sho", 2, 96, 700, 2000),
        # interpolation and forecast at test times
        _case("predict", "predict", "sho", 1, 33, 500, 2001, stars=400),
        # quasi-periodic product kernel
        _case("product_grad", "grad", "prod+m32", 0, 150, 500, 5000),
        # the FP64 filter that FP32 results are checked against
        _case("fp64_loglik", "loglik", "sho+m32", 1, 150, 300, 2500, precision=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: the same calls, with other sizes, kernels,
    instruments and dampings."""
    call = rng.choice(["loglik", "loglik", "long", "grad", "grad", "host", "graph", "fit",
                       "windows", "condition", "predict", "product", "fp64"])
    low_q = rng.random() < 0.15
    terms = rng.choice(["sho", "sho+m32", "sho+sho"])
    slots = rng.choice([0, 1, 1, 2, 3])
    layout = int(terms == "sho+sho" and slots == 1 and rng.random() < 0.5)
    if call == "long":
        n = _log(rng, 1000, 1 << 20)
        return _case(None, "loglik", terms, slots, 1, n, n, layout=layout, low_q=low_q)
    if call == "graph":
        n = _log(rng, 500, 100000)
        sets = _log(rng, 2, max(2, min(512, 4_000_000 // n)))
        return _case(None, call, terms, slots, 1, n, n, sets=sets, layout=layout, low_q=low_q)
    if call == "product":
        hi = _log(rng, 500, 10000)
        return _case(None, rng.choice(["loglik", "grad"]), rng.choice(["prod", "prod+m32"]), 0,
                     _log(rng, 1, 1_000_000 // hi), max(2, hi // 10), hi, low_q=low_q)
    if call == "fp64":
        hi = _log(rng, 50, 3000)
        return _case(None, "loglik", terms, slots, _log(rng, 1, 200), max(2, hi // 8), hi,
                     layout=layout, low_q=low_q, precision=64)
    if call in ("windows", "condition", "predict"):
        hi = _log(rng, 100, 2500)
        slots = max(slots, 1) if call == "windows" else slots
        return _case(None, call, terms, slots, _log(rng, 1, 200), max(2, hi // 5), hi,
                     layout=layout, low_q=low_q,
                     stars=_log(rng, 1, 2000) if call == "predict" else 0)
    hi = _log(rng, 100, 20000)
    most = 8_000_000 if call == "loglik" else 5_000_000
    return _case(None, call, terms, slots, _log(rng, 1, min(1024, most // hi)), max(2, hi // 10),
                 hi, layout=layout, low_q=low_q)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _lengths(case):
    """The same lengths for every seed, spread evenly over their logarithm."""
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    at = np.modf(0.5 + 0.6180339887498949 * np.arange(case["series"]))[0]
    return np.rint(np.exp(lo + (hi - lo) * at)).astype(np.int64)


def _theta(case, rng):
    centre = np.array(CENTRE[case["terms"]])
    quality = list(QUALITY[case["terms"]])
    if case["low_q"]:
        centre[quality] = 0.6
    if case["sets"]:
        th = centre * np.exp(0.5 * rng.standard_normal((case["sets"], len(centre))))
    else:
        th = centre * 10.0 ** rng.uniform(-0.5, 0.5, (case["series"], len(centre)))
    if not case["low_q"]:
        th[:, quality] = np.maximum(th[:, quality], 0.55)
    return np.concatenate([th, np.full((len(th), 1), WHITE)], axis=1).astype(np.float32)


def _tick(x):
    """Times are whole multiples of 2^-24, as of a clock: their sums are exact
    in FP64, so that the same seed gives the same times to the bit."""
    return torch.round(x * 2.0 ** 24) * 2.0 ** -24


def _running(x, first):
    """Cumulative sums of x that start anew at every index of ``first``."""
    c = torch.cumsum(x, 0)
    n = torch.diff(first, append=first.new_tensor([len(x)]))
    return c - torch.repeat_interleave(c[first] - x[first], n)


def _exposures(case, counts, g):
    """(t_start, t_end, instrument or None), in start order within each series."""
    dev, k = g.device, case["slots"]

    def unit(n):
        return torch.rand(n, generator=g, device=dev, dtype=torch.float64)

    def waits(n):  # Exp(1), never zero
        return _tick(-torch.log1p(-unit(n)) + 1e-6)

    n = int(counts.sum())
    if k <= 1:
        first = torch.as_tensor(np.cumsum(counts) - counts, device=dev)
        t = _running(waits(n), first)
        if k == 0:
            return t, t.clone(), None
        last = torch.as_tensor(np.cumsum(counts) - 1, device=dev)
        nxt = torch.cat([t[1:], t.new_tensor([math.inf])])
        nxt[last] = math.inf
        return t, torch.minimum(t + _tick(0.05 + 0.45 * unit(n)), nxt), None
    # instruments of their own cadence: exposure, dead time of the same mean
    if case["terms"] == "sho":
        lo, hi = np.full(k, 0.5), np.full(k, 3.0)
    else:
        lo = hi = np.array([0.1, 1.0, 5.0])[:k]
    share = 2.0 / (lo + hi)
    part = np.floor(counts[:, None] * (share / share.sum())).astype(np.int64)
    part[:, 0] += counts - part.sum(1)
    part = part.reshape(-1)
    keep = part > 0
    n_part = torch.as_tensor(part, device=dev)
    first = torch.as_tensor((np.cumsum(part) - part)[keep], device=dev)
    inst = torch.repeat_interleave(torch.arange(k, device=dev).repeat(len(counts)), n_part)
    lo_t, hi_t = torch.as_tensor(lo, device=dev)[inst], torch.as_tensor(hi, device=dev)[inst]
    dur = _tick(lo_t + (hi_t - lo_t) * unit(n))
    t_e = _running(dur + _tick(0.5 * (lo_t + hi_t) * waits(n)), first)
    t_s = t_e - dur
    sid = torch.repeat_interleave(torch.arange(len(counts), device=dev),
                                  torch.as_tensor(counts, device=dev))
    order = torch.argsort(sid * (2.0 * float(t_e.max()) + 1.0) + t_s, stable=True)
    return t_s[order], t_e[order], inst[order].to(torch.int32)


def _frequencies(w0, q, g, n):
    """n angular frequencies per row from the oscillator's power spectrum."""
    x = torch.logspace(-2, 2, 801, dtype=torch.float64, device=g.device)
    dens = 1.0 / ((x * x - 1.0) ** 2 + (x / q[:, None]) ** 2)
    cdf = torch.cumsum(0.5 * (dens[:, 1:] + dens[:, :-1]) * torch.diff(x), 1)
    u = torch.rand(len(w0), n, generator=g, device=g.device, dtype=torch.float64) * cdf[:, -1:]
    i = torch.searchsorted(cdf, u).clamp(max=len(x) - 2)
    return w0[:, None] * x[i]


def _draw_of(sig, w0, q, sid, mid, half, g, n=16):
    """Exposure averages of a random sum of cosines with that spectrum."""
    w = _frequencies(w0, q, g, n)
    ph = TWO_PI * torch.rand(len(w0), n, generator=g, device=g.device, dtype=torch.float64)
    out = torch.zeros_like(mid)
    for j in range(n):
        wj = w[sid, j]
        out += torch.cos(wj * mid + ph[sid, j]) * torch.sinc(wj * half / math.pi)
    return out * (sig * math.sqrt(2.0 / n))[sid]


def _data(case, seed):
    rng = np.random.default_rng(seed)
    counts = _lengths(case)
    theta = _theta(case, rng)
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(int(rng.integers(1 << 62)))
    t_s, t_e, inst = _exposures(case, counts, g)
    sid = torch.repeat_interleave(torch.arange(len(counts), device=dev),
                                  torch.as_tensor(counts, device=dev))
    rows = (np.tile(np.append(CENTRE[case["terms"]], WHITE), (len(counts), 1))
            if case["sets"] else theta)
    p = torch.as_tensor(rows, dtype=torch.float64, device=dev)
    mid, half = 0.5 * (t_s + t_e), 0.5 * (t_e - t_s)
    y = torch.zeros_like(mid)
    j = 0
    for kind in TERMS[case["terms"]]:
        if kind == gp.SHO_PRODUCT:
            one = torch.ones_like(p[:, j])
            y += (_draw_of(one, p[:, j + 1], p[:, j + 2], sid, mid, half, g) *
                  _draw_of(p[:, j], p[:, j + 3], p[:, j + 4], sid, mid, half, g))
            j += 5
        elif kind == gp.SHO:
            y += _draw_of(p[:, j], p[:, j + 1], p[:, j + 2], sid, mid, half, g)
            j += 3
        else:
            y += _draw_of(p[:, j], math.sqrt(3.0) / p[:, j + 1],
                          torch.full_like(p[:, j], 0.5), sid, mid, half, g)
            j += 2
    n = len(y)
    y += WHITE * torch.randn(n, generator=g, device=dev, dtype=torch.float64)
    yerr = 0.02 + 0.08 * torch.rand(n, generator=g, device=dev, dtype=torch.float64)
    data = {"offsets": np.concatenate([[0], np.cumsum(counts)]).astype(np.int64),
            "t_s": t_s, "t_e": t_e, "inst": inst, "y": y.float(), "yerr": yerr.float(),
            "theta": theta}
    if case["stars"]:
        a, b = data["offsets"][:-1], data["offsets"][1:] - 1
        t0, t1 = t_s.cpu().numpy()[a] - 2.0, t_e.cpu().numpy()[b] + 10.0
        data["stars"] = np.sort(rng.uniform(t0[:, None], t1[:, None],
                                            (len(counts), case["stars"])), 1).reshape(-1)
    return data


def prepare(case, seed):
    d = _data(case, seed)
    inst = None if d["inst"] is None else d["inst"].cpu().numpy()
    model = gp.Model(TERMS[case["terms"]], d["offsets"], d["t_s"].cpu().numpy(),
                     d["t_e"].cpu().numpy(), d["y"].cpu().numpy(), d["yerr"].cpu().numpy(), inst,
                     layout=case["layout"], precision=case["precision"])
    theta = torch.as_tensor(d["theta"], device=_device())
    state = {"call": case["call"], "model": model, "theta": theta,
             "per_series": not case["sets"]}
    if case["call"] == "host":
        state["theta"] = d["theta"]
    elif case["call"] == "fit":
        theta.requires_grad_(True)
    elif case["call"] == "graph":  # a graph replays on fixed buffers
        rows = model.n_out(theta, state["per_series"])
        state["out"] = torch.empty(rows, dtype=torch.float64, device=theta.device)
        state["grad"] = torch.empty(rows, model.n_params, dtype=torch.float32,
                                    device=theta.device)
    elif case["call"] == "predict":
        state["stars"] = d["stars"]
        state["star_offsets"] = case["stars"] * np.arange(case["series"] + 1, dtype=np.int64)
    return state


def run(state):
    call, model, theta, ps = (state[k] for k in ("call", "model", "theta", "per_series"))
    if call == "loglik":
        return {"ll": model.loglik(theta, per_series=ps)}
    if call == "grad":
        ll, grad = model.loglik_grad(theta, per_series=ps)
        return {"ll": ll, "grad": grad}
    if call == "graph":
        ll, grad = model.loglik_grad(theta, per_series=ps, out=state["out"], grad=state["grad"],
                                     batched=True)
        return {"ll": ll, "grad": grad}
    if call == "host":
        ll, grad = model.loglik_grad_host(theta, per_series=ps, reupload_events=True)
        return {"ll": ll, "grad": grad}
    if call == "fit":
        theta.grad = None
        ll = gp.loglik(model, theta, per_series=ps)
        ll.sum().backward()
        return {"ll": ll.detach(), "grad": theta.grad}
    if call == "windows":
        ll, grad, dexp = model.loglik_grad(theta, per_series=ps, exposure=True)
        return {"ll": ll, "grad": grad, "windows": dexp}
    if call == "condition":
        ll, cond = model.condition(theta, per_series=ps)
        return {"ll": ll, "mean": cond[..., 0], "var": cond[..., 1]}
    ll, pred = model.predict(theta, state["stars"], state["star_offsets"], per_series=ps)
    return {"ll": ll, "mean": pred[..., 0], "var": pred[..., 1]}


def work(case):
    """Bytes of the event stream (per exposure two gaps, two tags, y, yerr^2
    and 1/length; per instant one gap, tag, y and yerr^2), the parameters and
    the outputs; operations of the filter with its structure used: per event
    and parameter vector a predicted covariance and the step's scalars, per
    measurement one update, and twice as much again for a reverse sweep."""
    lo, hi = case["n_min"], case["n_max"]
    mean = lo if lo == hi else (hi - lo) / math.log(hi / lo)
    n, rep = mean * case["series"], max(1, case["sets"])
    n_params = len(CENTRE[case["terms"]]) + 1
    d = {"sho": 2, "sho+m32": 4, "sho+sho": 4, "prod": 4, "prod+m32": 6}[case["terms"]]
    n_osc = {"sho": 1, "sho+m32": 2, "sho+sho": 2, "prod": 2, "prod+m32": 3}[case["terms"]]
    out_rows = case["series"] * rep
    events = 1 if case["slots"] == 0 else 2
    dz = d + case["slots"]
    predict = (4 * d ** 3 if "prod" in case["terms"] else 6 * d * dz) + 60 * n_osc
    update = 1.5 * dz * (dz + 1) + 10
    flops = n * rep * (events * predict + update)
    size = n * (13 if case["slots"] == 0 else 22) + 4 * n_params * (case["sets"] or
                                                                    case["series"])
    size += 8 * out_rows
    if case["call"] in ("grad", "graph", "host", "fit", "windows"):
        flops *= 3
        size += 4 * n_params * out_rows
    if case["call"] in ("windows", "condition"):
        flops *= 1 if case["call"] == "windows" else 3
        size += 8 * n * rep
    if case["call"] == "predict":
        flops *= 3
        size += 16 * case["stars"] * out_rows
    return {"bytes": float(size), "flops": float(flops)}


# ---------------------------------------------------------------------------
# The same results in 64 bits: a sequential filter in plain torch, every row
# (a stretch of one series under one parameter vector) a batch entry.
# ---------------------------------------------------------------------------
def _oscillators(case, th):
    """Per oscillator (a, beta, w2, variance), columns over rows; th [R, np]."""
    out, j = [], 0
    one = torch.ones_like(th[:, 0])
    for kind in TERMS[case["terms"]]:
        if kind == gp.SHO_PRODUCT:
            pars = [(one, th[:, j + 1], th[:, j + 2]), (th[:, j], th[:, j + 3], th[:, j + 4])]
            j += 5
        elif kind == gp.SHO:
            pars = [(th[:, j], th[:, j + 1], th[:, j + 2])]
            j += 3
        else:
            pars = [(th[:, j], math.sqrt(3.0) / th[:, j + 1], 0.5 * one)]
            j += 2
        for sig, w0, q in pars:
            a = w0 / (2.0 * q)
            out.append((a, torch.where(q == 0.5, 0.0 * a, w0 * w0 - a * a), w0 * w0, sig * sig))
    return out


def _impulse(t, a, beta):
    """f(t) = e^{-a t} sin(b t)/b and f'(t), b = sqrt(beta) (any sign of beta)."""
    b = torch.sqrt(torch.where(beta == 0, torch.ones_like(beta), beta.abs()))
    e = torch.exp(-a * t)
    s_u, c_u = e * torch.sin(b * t) / b, e * torch.cos(b * t)
    b_o = torch.where(beta < 0, b, torch.zeros_like(b))  # b < a here
    e1, e2 = torch.exp((b_o - a) * t), torch.exp(-(a + b_o) * t)
    f = torch.where(beta > 0, s_u, torch.where(beta < 0, 0.5 * (e1 - e2) / b, e * t))
    c = torch.where(beta > 0, c_u, torch.where(beta < 0, 0.5 * (e1 + e2), e))
    return f, c - a * f


def _series(a, w2):
    """Taylor coefficients in t, per oscillator [..., R], of f/t, f', F1/t^2,
    I_ff/t^3, I_pp/t and I_FF/t^5, from f'' + 2 a f' + w2 f = 0."""
    N = 20
    c = [torch.zeros_like(a), torch.ones_like(a)]
    for n in range(N):
        c.append(-(2 * a * (n + 1) * c[n + 1] + w2 * c[n]) / ((n + 2) * (n + 1)))
    out = [[] for _ in range(6)]
    for k in range(N - 2):
        out[0].append(c[k + 1])
        out[1].append((k + 1) * c[k + 1])
        out[2].append(c[k + 1] / (k + 2))
        pairs = [(n, k + 2 - n) for n in range(1, k + 2)]
        out[3].append(sum(c[n] * c[m] for n, m in pairs) / (k + 3))
        out[4].append(sum(n * m * c[n] * c[m] for n, m in pairs) / (k + 1))
        out[5].append(sum(c[n] * c[m] / ((n + 1) * (m + 1)) for n, m in pairs) / (k + 5))
    return out


def _scalars(t, a, beta, w2):
    """f, f', F1 = int f, and the integrals of f^2, f'^2 and F1^2 over [0, t]:
    closed forms, or series where those cancel."""
    f, fp = _impulse(t, a, beta)
    F1 = (1 - fp - 2 * a * f) / w2
    Ipp = (1 - fp * fp - w2 * f * f) / (4 * a)
    Iff = (Ipp - f * fp - a * f * f) / w2
    IFF = (t + Ipp + 4 * a * a * Iff - 2 * f - 4 * a * F1 + 2 * a * f * f) / (w2 * w2)
    rate = torch.maximum(torch.sqrt(w2), 2 * a)
    small = rate * t < 0.6
    ts = torch.where(small, t, torch.zeros_like(t))
    out = []
    for x, coeffs, power in zip((f, fp, F1, Iff, Ipp, IFF), _series(a, w2), (1, 0, 2, 3, 1, 5)):
        acc = coeffs[-1]
        for g in reversed(coeffs[:-1]):
            acc = acc * ts + g
        out.append(torch.where(small, acc * ts ** power, x))
    return out


def _mat(rows):
    return torch.stack([torch.stack(r, -1) for r in rows], -2)


def _step_matrices(case, osc, t):
    """Phi, Q [..., D, D] for gaps t [..., R]: latent states, then one integral
    state per slot that integrates the latent."""
    blocks = []
    for a, beta, w2, var in osc:
        sc = _scalars(t, a, beta, w2)
        f, fp = sc[:2]
        phi = [[fp + 2 * a * f, f], [-w2 * f, fp]]
        p_inf = torch.diag_embed(torch.stack([var, var * w2], -1))
        blocks.append((phi, p_inf, sc))
    if case["terms"].startswith("prod"):
        pa, pb = _mat(blocks[0][0]), _mat(blocks[1][0])
        phi = (pa[..., :, None, :, None] * pb[..., None, :, None, :]).flatten(-2).flatten(-3, -2)
        p0 = (blocks[0][1][..., :, None, :, None] *
              blocks[1][1][..., None, :, None, :]).flatten(-2).flatten(-3, -2)
        q = p0 - phi @ p0 @ phi.mT
        if len(blocks) == 3:
            pc, c0 = _mat(blocks[2][0]), blocks[2][1]
            phi, q = _block_diag(phi, pc), _block_diag(q, c0 - pc @ c0 @ pc.mT)
            p0 = _block_diag(p0, c0)
        return phi, q, p0
    d, ns = 2 * len(osc), case["slots"]
    zero, one = torch.zeros_like(t), torch.ones_like(t)
    P = [[zero] * (d + ns) for _ in range(d + ns)]
    Q = [[zero] * (d + ns) for _ in range(d + ns)]
    qzz = zero
    p0 = []
    for i, ((a, beta, w2, var), (phi, _, (f, fp, F1, Iff, Ipp, IFF))) in enumerate(
            zip(osc, blocks)):
        qc = 4.0 * a * w2 * var
        x, v = 2 * i, 2 * i + 1
        P[x][x], P[x][v], P[v][x], P[v][v] = phi[0][0], phi[0][1], phi[1][0], phi[1][1]
        Q[x][x], Q[v][v] = qc * Iff, qc * Ipp
        Q[x][v] = Q[v][x] = 0.5 * qc * f * f
        qzz = qzz + qc * IFF
        for z in range(d, d + ns):
            P[z][x], P[z][v] = f + 2 * a * F1, F1
            Q[z][x] = Q[x][z] = 0.5 * qc * F1 * F1
            Q[z][v] = Q[v][z] = qc * (f * F1 - Iff)
        p0 += [var, var * w2]
    for z in range(d, d + ns):
        P[z][z] = one
        for z2 in range(d, d + ns):
            Q[z][z2] = qzz
        p0.append(torch.ones_like(p0[0]))
    return _mat(P), _mat(Q), torch.diag_embed(torch.stack(p0, -1))


def _block_diag(x, y):
    shape = torch.broadcast_shapes(x.shape[:-2], y.shape[:-2])
    x, y = x.expand(*shape, *x.shape[-2:]), y.expand(*shape, *y.shape[-2:])
    n, m = x.shape[-1], y.shape[-1]
    return torch.cat([torch.cat([x, x.new_zeros(*shape, n, m)], -1),
                      torch.cat([y.new_zeros(*shape, m, n), y], -1)], -2)


_END, _INSTANT, _START, _STAR = 0, 1, 2, 3


def _events(case, d):
    """Per event, series by series in time order: kind, source index (a
    measurement, or a test time); and the series' event offsets."""
    dev = d["t_s"].device
    counts = torch.as_tensor(np.diff(d["offsets"]), device=dev)
    sid = torch.repeat_interleave(torch.arange(len(counts), device=dev), counts)
    n = len(sid)
    src = torch.arange(n, device=dev)
    if case["slots"] == 0:
        parts = [(d["t_s"], _INSTANT, src, sid)]
    else:
        parts = [(d["t_s"], _START, src, sid), (d["t_e"], _END, src, sid)]
    if case["stars"]:
        t = torch.as_tensor(d["stars"], device=dev)
        parts.append((t, _STAR, torch.arange(len(t), device=dev),
                      torch.arange(len(counts), device=dev).repeat_interleave(case["stars"])))
    t = torch.cat([p[0] for p in parts])
    kind = torch.cat([torch.full_like(p[2], p[1]) for p in parts])
    src, sid = torch.cat([p[2] for p in parts]), torch.cat([p[3] for p in parts])
    order = torch.arange(len(t), device=dev)
    for key in (kind, t, sid):  # stable sorts, the last key first in rank
        order = order[torch.argsort(key[order], stable=True)]
    off = torch.cumsum(torch.bincount(sid, minlength=len(counts)), 0).cpu().numpy()
    return kind[order], src[order], np.concatenate([[0], off])


def _filter(case, d, ev, first, count, last, theta, star=None):
    """Log-likelihood per row r: events [first, last) of the stream, those from
    ``count`` on counted, under theta[r].  d's t_s, t_e, y and R (noise
    variances [R or 1, N]) may need gradients.  star = (eps, kap), zeros
    [steps, R]: also returns the latent's mean and variance at test times, and
    shifts the state by eps P h and kap P h h^T P there."""
    kind, src, _ = ev
    dev = theta.device
    R = len(first)
    osc = _oscillators(case, theta)
    _, _, p0 = _step_matrices(case, osc, torch.ones(R, dtype=torch.float64, device=dev))
    D, ns = p0.shape[-1], case["slots"]
    lat = torch.zeros(D, dtype=torch.float64, device=dev)
    if case["terms"].startswith("prod"):
        lat[0:D:4] = 1.0
    else:
        lat[0:D - ns:2] = 1.0
    is_start, is_star = kind == _START, kind == _STAR
    times = torch.where(is_start | (kind == _INSTANT), d["t_s"][src.clamp(max=len(d["t_s"]) - 1)],
                        d["t_e"][src.clamp(max=len(d["t_e"]) - 1)])
    if case["stars"]:
        stars = torch.as_tensor(d["stars"], device=dev)
        times = torch.where(is_star, stars[src.clamp(max=len(stars) - 1)], times)
    slot = (torch.zeros_like(src) if d["inst"] is None
            else d["inst"].to(torch.int64)[src.clamp(max=len(d["t_s"]) - 1)])
    P, m = p0.expand(R, D, D).clone(), p0.new_zeros(R, D, 1)
    white = theta[:, -1] ** 2
    steps = int((last - first).max())
    block = max(1, min(steps, int(1.5e8 // (R * D * D))))
    ll = torch.zeros(R, dtype=torch.float64, device=dev)
    seen = []
    for k0 in range(0, steps, block):
        k = torch.arange(k0, min(k0 + block, steps), device=dev)[:, None]
        e = first[None, :] + k
        live = e < last[None, :]
        e = torch.where(live, e, first[None, :])
        gap = torch.where(live & (k > 0), times[e] - times[(e - 1).clamp(min=0)],
                          torch.zeros((), dtype=torch.float64, device=dev))
        Phi, Q, _ = _step_matrices(case, osc, gap)
        st = live & is_start[e]
        reads = live & (kind[e] <= _INSTANT)
        i = src[e].clamp(max=len(d["y"]) - 1)
        if ns:
            hot = torch.nn.functional.one_hot(slot[e], ns).to(torch.float64)
            keep = torch.cat([torch.ones(*e.shape, D - ns, dtype=torch.float64, device=dev),
                              1 - hot * st[..., None]], -1)
            Phi, Q = Phi * keep[..., None], Q * keep[..., None] * keep[..., None, :]
            w = 1.0 / torch.where(reads, d["t_e"][i] - d["t_s"][i], torch.ones_like(gap))
            h = torch.cat([torch.zeros(*e.shape, D - ns, dtype=torch.float64, device=dev),
                           hot * w[..., None]], -1)
        else:
            h = lat.expand(*e.shape, D)
        h = (h * reads[..., None])[..., None]
        noise = torch.where(reads, d["R"][i] + white, torch.ones_like(gap))
        y = torch.where(reads, d["y"][i], torch.zeros_like(gap))
        PhiT, act = Phi.mT.contiguous(), reads.to(torch.float64)
        S_all, v_all = [], []
        for j in range(len(k)):
            T = Phi[j] @ torch.cat([P, m], -1)
            P = torch.baddbmm(Q[j], T[..., :D], PhiT[j])
            m = T[..., D:]
            if star is not None:
                on = is_star[e[j]] & live[j]
                u = P @ lat[:, None]
                seen.append((on, e[j], (lat @ m)[:, 0], (lat @ u)[:, 0]))
                go = torch.where(on, star[0][k0 + j], torch.zeros_like(star[0][k0 + j]))
                gk = torch.where(on, star[1][k0 + j], torch.zeros_like(star[1][k0 + j]))
                m = m + go[:, None, None] * u
                P = P + gk[:, None, None] * (u @ u.mT)
            u = P @ h[j]
            S = (h[j] * u).sum((1, 2)) + noise[j]
            v = y[j] - (h[j] * m).sum((1, 2))
            iS = (act[j] / S)[:, None, None]
            m = m + u * (v[:, None, None] * iS)
            P = P - (u * iS) @ u.mT
            S_all.append(S)
            v_all.append(v)
        S, v = torch.stack(S_all), torch.stack(v_all)
        counted = (reads & (e >= count[None, :])).to(torch.float64)
        ll = ll - 0.5 * (counted * (torch.log(TWO_PI * S) + v * v / S)).sum(0)
    return (ll, seen) if star is not None else ll


# a stretch counts STRETCH events after BURN more that only bring its state to
# what the series' whole past would have left (their influence decays within
# a few hundred events)
STRETCH, BURN = 8000, 4000


def _exact_ll(case, d, ev, theta_rows, series_of):
    """Log-likelihood per (parameter vector, series) pair."""
    off, dev = ev[2], d["t_s"].device
    row, a, c, b = [], [], [], []
    for r, s in enumerate(series_of):
        for k in range(off[s], max(off[s + 1], off[s] + 1), STRETCH):
            row.append(r)
            a.append(max(off[s], k - BURN))
            c.append(k)
            b.append(min(off[s + 1], k + STRETCH))
    row, a, c, b = (torch.as_tensor(np.array(x, dtype=np.int64), device=dev)
                    for x in (row, a, c, b))
    ll = torch.zeros(len(series_of), dtype=torch.float64, device=dev)
    with torch.no_grad():
        for g in torch.split(torch.argsort(b - a, descending=True, stable=True), 150_000):
            ll.index_add_(0, row[g], _filter(case, d, ev, a[g], c[g], b[g], theta_rows[row[g]]))
    return ll


def exact(case, seed):
    d = _data(case, seed)
    dev = d["t_s"].device
    theta = torch.as_tensor(d["theta"], device=dev).double()
    d["y"], d["R"] = d["y"].double(), d["yerr"].double() ** 2
    ev = _events(case, d)
    S, rows = case["series"], len(theta)
    call = case["call"]
    if call in ("loglik", "grad", "graph", "host", "fit"):
        pick, series = ((np.arange(S), np.arange(S)) if not case["sets"] else
                        (np.repeat(np.arange(rows), S), np.tile(np.arange(S), rows)))
        variants = [torch.zeros_like(theta[0])]
        step = 2e-4
        if call != "loglik":  # fourth-order differences of relative steps
            for p in range(theta.shape[1]):
                for m in (-2, -1, 1, 2):
                    variants.append(torch.zeros_like(theta[0]).index_fill_(
                        0, torch.tensor([p], device=dev), m * step))
        th = torch.cat([theta[pick] * (1 + v) for v in variants])
        ll = _exact_ll(case, d, ev, th, np.tile(series, len(variants))).view(len(variants), -1)
        if call == "loglik":
            return {"ll": ll[0]}
        f = ll[1:].view(-1, 4, len(pick))
        g = ((8 * (f[:, 2] - f[:, 1]) - (f[:, 3] - f[:, 0])) / (12 * step)).T / theta[pick]
        if call == "fit" and case["sets"]:
            g = g.view(rows, S, -1).sum(1)
        return {"ll": ll[0], "grad": g}
    # one row per series (these calls are drawn with a vector per series)
    off = torch.as_tensor(ev[2], device=dev)
    first, last = off[:-1], off[1:]
    leaves = {k: d[k].clone().requires_grad_(True) for k in ("t_s", "t_e", "y", "R")}
    theta.requires_grad_(True)
    if call == "predict":
        zero = torch.zeros(int((last - first).max()), S, dtype=torch.float64, device=dev)
        eps, kap = zero.clone().requires_grad_(True), zero.clone().requires_grad_(True)
        ll, seen = _filter(case, d, ev, first, first, last, theta, star=(eps, kap))
        g_e, g_k = torch.autograd.grad(ll.sum(), (eps, kap))
        on, e, hm, hu = (torch.stack(x) for x in zip(*seen))
        at = ev[1][e[on]]
        mean = torch.zeros(len(d["stars"]), dtype=torch.float64, device=dev)
        var = mean.clone()
        mean[at] = (hm + g_e)[on].detach()
        var[at] = (hu + 2 * g_k - g_e * g_e)[on].detach()
        return {"ll": ll.detach(), "mean": mean[None], "var": var[None]}
    ll = _filter(case, {**d, **leaves}, ev, first, first, last, theta)
    if call == "windows":
        g_s, g_e, g_t = torch.autograd.grad(ll.sum(), (leaves["t_s"], leaves["t_e"], theta))
        return {"ll": ll.detach(), "grad": g_t, "windows": torch.stack([g_s, g_e], -1)[None]}
    # the data's influence gives the conditioned values: with alpha = K^-1 y =
    # -dL/dy and (K^-1)_nn = alpha^2 - 2 dL/dR, mean = y - R alpha and
    # var = R - R^2 (K^-1)_nn
    g_y, g_r = torch.autograd.grad(ll.sum(), (leaves["y"], leaves["R"]))
    sid = torch.repeat_interleave(torch.arange(S, device=dev),
                                  torch.as_tensor(np.diff(d["offsets"]), device=dev))
    noise = (d["R"] + theta.detach()[sid, -1] ** 2)
    mean = d["y"] + noise * g_y
    var = noise - noise ** 2 * (g_y ** 2 - 2 * g_r)
    return {"ll": ll.detach(), "mean": mean[None], "var": var[None]}
