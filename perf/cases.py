"""What this library is measured on: its public entry points over the range of
calls that its users make.

Orders and arguments are those of the repository's own workloads: the paper's
sweep (v = 2^0 .. 2^10, x uniform in [1, 100]), its Small region ([0, 150]^2),
the robustness sweep (v and x log-uniform to 1e5) and von Mises-Fisher
concentrations in high dimension.  Calls go from one pair to tens of millions,
in both data types, with one order per call and one per pair, values and
x-derivatives, on device tensors, host buffers and through the server.
"""
import math

import numpy as np
import torch

import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import vmf
from paper_2409_08729_gb300.serve import Server

SWEEP = [float(2 ** k) for k in range(11)]
DIMS = (2048, 8192, 32768)
_server = None


def listed():
    return [
        # the smallest call there is: one pair, as a fit or a sampler's accept step makes it
        {"name": "one_pair_k", "op": "log_k", "dtype": "f64", "orders": "one", "v": 2.5, "x": "small", "n": 1},
        # a few hundred points of a plot or a table, an order each, not a multiple of anything
        {"name": "points_i", "op": "log_i", "dtype": "f64", "orders": "small", "v": 0.0, "x": "small", "n": 997},
        # the plain configuration: 11 orders with 10,000 arguments each in one call
        {"name": "plain_k", "op": "log_k", "dtype": "f64", "orders": "sweep", "v": 0.0, "x": "sweep", "n": 110000},
        # the paper's sweep, one order per call (a kernel density, a Matern covariance): 20M arguments
        {"name": "sweep_i_order", "op": "log_i", "dtype": "f64", "orders": "one", "v": 8.0, "x": "sweep",
         "n": 20000000},
        # the paper's sweep, an order per pair
        {"name": "sweep_k_mixed", "op": "log_k", "dtype": "f64", "orders": "sweep", "v": 0.0, "x": "sweep",
         "n": 22000000},
        # orders and arguments over the whole domain, the costliest mix
        {"name": "robust_k", "op": "log_k", "dtype": "f64", "orders": "robust", "v": 0.0, "x": "robust",
         "n": 16000001},
        # single precision, the paper's sweep with an order per pair
        {"name": "sweep_i_f32", "op": "log_i", "dtype": "f32", "orders": "sweep", "v": 0.0, "x": "sweep",
         "n": 24000000},
        # single precision over the whole domain
        {"name": "robust_k_f32", "op": "log_k", "dtype": "f32", "orders": "robust", "v": 0.0, "x": "robust",
         "n": 16000001},
        # a training step's two directions: values, and the gradient in x by autograd
        {"name": "grad_k", "op": "grad_k", "dtype": "f64", "orders": "sweep", "v": 0.0, "x": "sweep", "n": 4000003},
        # the vMF log-normaliser of a batch of concentrations and its derivative (d/2 - 1 = 1023)
        {"name": "vmf_log_c", "op": "vmf", "dtype": "f64", "orders": "one", "v": 2048.0, "x": "kappa", "n": 1000001},
        # end to end on pinned host buffers
        {"name": "host_k", "op": "host_k", "dtype": "f64", "orders": "sweep", "v": 0.0, "x": "sweep", "n": 8000000},
        # the serving mix: requests of uneven sizes, half log I, 70 % single precision, on device buffers
        {"name": "served", "op": "served", "dtype": "mixed", "orders": "robust", "v": 0.0, "x": "robust", "n": 2000000,
         "requests": 96},
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1


def draw(rng):
    op = rng.choice(["log_i", "log_k", "log_i", "log_k", "log_i_dx", "log_k_dx", "grad_i", "grad_k", "vmf", "host_i",
                     "host_k", "served"])
    if op == "vmf":
        return {"op": op, "dtype": "f64", "orders": "one", "v": float(rng.choice(DIMS)), "x": "kappa",
                "n": _log_size(rng, 1, 8000000)}
    if op == "served":
        n = _log_size(rng, 20000, 2000000)
        return {"op": op, "dtype": "mixed", "orders": "robust", "v": 0.0, "x": "robust", "n": n,
                "requests": rng.randint(8, 96)}
    dtype = rng.choice(["f64", "f32"]) if op in ("log_i", "log_k", "host_i", "host_k") else "f64"
    orders = rng.choice(["one", "sweep", "small", "robust"])
    x = {"one": rng.choice(["sweep", "robust"]), "sweep": "sweep", "small": "small", "robust": "robust"}[orders]
    v = 0.0
    if orders == "one":
        v = rng.choice([0.0, 0.5, round(math.exp(rng.uniform(math.log(0.1), math.log(2000.0))), 6)])
    n = _log_size(rng, 1, 8000000 if "k" in op else 12000000)
    return {"op": op, "dtype": dtype, "orders": orders, "v": v, "x": x, "n": n}


def _loguniform(n, lo, hi, g):
    t = torch.empty(n, dtype=torch.float64, device="cuda")
    return t.uniform_(math.log(lo), math.log(hi), generator=g).exp_()


def _pairs(orders, xdist, v0, n, g, vmax=1e5, xmin=1e-6, xmax=1e5):
    """(v, x) on the device in double precision; v is None for one order."""
    v = None
    if orders == "sweep":
        idx = torch.randint(0, len(SWEEP), (n,), generator=g, device="cuda")
        v = torch.tensor(SWEEP, dtype=torch.float64, device="cuda")[idx]
    elif orders == "small":
        v = torch.empty(n, dtype=torch.float64, device="cuda").uniform_(0.0, 150.0, generator=g)
    elif orders == "robust":
        # 1 % exactly zero, 1 % exactly one half
        v = _loguniform(n, 1e-6, vmax, g)
        u = torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
        v[u < 0.01] = 0.0
        v[(u >= 0.01) & (u < 0.02)] = 0.5
    if xdist == "robust":
        x = _loguniform(n, xmin, xmax, g)
    elif xdist == "kappa":
        x = _loguniform(n, 0.1 * v0, 10.0 * v0, g)
    else:
        lo, hi = (1.0, 100.0) if xdist == "sweep" else (0.0, 150.0)
        x = torch.empty(n, dtype=torch.float64, device="cuda").uniform_(lo, hi, generator=g)
        x.clamp_(min=1e-9)
    return v, x


def _sizes(case):
    """Sizes (log-uniform, about n in all), kinds and types of the serving
    mix's requests: the case's own, the same for every seed."""
    r = np.random.default_rng(case["n"] * 7919 + case["requests"])
    w = np.exp(r.uniform(0.0, math.log(2000.0), case["requests"]))
    s = np.maximum(1, (w * (case["n"] / w.sum())).astype(np.int64))
    return s, r.random(case["requests"]) < 0.5, r.random(case["requests"]) < 0.7


def _inputs(case, seed):
    """The inputs of a case: (v, x) in double precision at the values the call
    sees (rounded to single precision where it takes that), or one such pair
    per request with its kind and type."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["op"] != "served":
        v, x = _pairs(case["orders"], case["x"], case["v"], case["n"], g)
        if v is None:
            v = torch.tensor([case["v"]], dtype=torch.float64, device="cuda")
        dt = torch.float32 if case["dtype"] == "f32" else torch.float64
        return v.to(dt), x.to(dt)
    reqs = []
    for n, is_i, single in zip(*_sizes(case)):
        v, x = _pairs("robust", "robust", 0.0, int(n), g, vmax=1e4, xmin=1e-3, xmax=1e4)
        dt = torch.float32 if single else torch.float64
        reqs.append(("i" if is_i else "k", v.to(dt), x.to(dt)))
    return reqs


def _the_server():
    # one server for the life of the process, as a serving program keeps it
    global _server
    if _server is None:
        _server = Server(arena_bytes=1 << 30, max_slots=256, ctas_per_sm=4, idle_ms=0.5)
    return _server


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "d": case["v"]}
    if op == "served":
        s["server"] = _the_server()
        s["reqs"] = [(k, v, x, torch.empty_like(x)) for k, v, x in _inputs(case, seed)]
        return s
    s["v"], s["x"] = _inputs(case, seed)
    if op.startswith("grad"):
        s["x"].requires_grad_(True)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        s["g"] = torch.empty_like(s["v"] if s["v"].numel() == s["x"].numel() else s["x"]).uniform_(-1, 1, generator=g)
    elif op.startswith("host"):
        for k in ("v", "x"):
            h = torch.empty(s[k].shape, dtype=s[k].dtype, pin_memory=True)
            s[k] = h.copy_(s[k])
        s["out"] = torch.empty(s["x"].shape, dtype=s["x"].dtype, pin_memory=True)
    return s


def run(state):
    op = state["op"]
    if op == "served":
        srv = state["server"]
        tickets = [srv.submit_device(k, v, x, out, ready=None) for k, v, x, out in state["reqs"]]
        for t in tickets:
            srv.wait(t)
            srv.release(t)
        return [torch.cat([out for _, _, x, out in state["reqs"] if x.dtype == dt] or
                          [torch.empty(0, dtype=dt, device="cuda")]) for dt in (torch.float64, torch.float32)]
    v, x = state["v"], state["x"]
    if op == "vmf":
        return vmf.log_c(state["d"], x), vmf.log_c(state["d"], x, deriv=True)
    if op.startswith("host"):
        return lb.host_eval("log_i" if op == "host_i" else "log_k", v, x, out=state["out"])
    if op.startswith("grad"):
        y = (lb.log_i if op == "grad_i" else lb.log_k)(v, x)
        return y.detach(), torch.autograd.grad(y, x, state["g"])[0]
    return getattr(lb, op)(v, x)


def work(case):
    """Each argument (and order, where every pair has its own) read once and
    each result written once; about 30 operations per value and 40 per
    derivative (a dozen terms of an expansion and two elementary functions)."""
    n, size = case["n"], 4 if case["dtype"] == "f32" else 8
    per_order = 0 if case["orders"] == "one" else size
    op = case["op"]
    if op == "served":
        return {"bytes": n * (0.7 * 12 + 0.3 * 24), "flops": 30.0 * n}
    if op == "vmf":
        return {"bytes": 3.0 * 8 * n, "flops": 70.0 * n}
    if op.startswith("grad"):
        return {"bytes": float(n * (4 * 8 + per_order)), "flops": 70.0 * n}
    return {"bytes": float(n * (2 * size + per_order)), "flops": (40.0 if op.endswith("dx") else 30.0) * n}


# Values in 64 bits by other means than the library's: the integral
# K_v = int_0^inf exp(-x cosh t) cosh(v t) dt by the trapezoid rule about its
# maximum; I_v by its power series, or, for v^2 + x^2 > 3600, by the trapezoid
# rule along the path of steepest descent of its contour integral.

def _plain_k(v, x, deriv):
    v = v.abs()[:, None]
    x = x[:, None]
    r = torch.hypot(v, x)
    t0 = torch.asinh(v / x)

    a = 0.5 * (r + v)
    b = 0.25 * x * x / a

    def drop(d):                                   # exponent below its maximum at t0 + d
        return a * (torch.expm1(d) - d) + b * (torch.expm1(-d) + d)

    lo, hi = torch.zeros_like(x), t0.clone()
    for _ in range(40):
        m = 0.5 * (lo + hi)
        big = drop(-m) > 42.0
        lo, hi = torch.where(big, lo, m), torch.where(big, m, hi)
    left = torch.where(drop(-t0) > 42.0, hi, t0)
    lo, hi = torch.zeros_like(x), torch.full_like(x, 60.0)
    for _ in range(40):
        m = 0.5 * (lo + hi)
        big = drop(m) > 42.0
        lo, hi = torch.where(big, lo, m), torch.where(big, m, hi)
    k = 192
    h = (left + hi) / k
    j = torch.arange(k + 1, dtype=torch.float64, device=x.device)[None]
    d = h * j - left
    t = (t0 + d).clamp_(min=0.0)
    w = torch.exp(-drop(d)) * (0.5 + 0.5 * torch.exp(-2 * v * t))
    w[:, 0] *= 0.5
    s = w.sum(1, keepdim=True)
    if deriv:
        return (-(w * torch.cosh(t)).sum(1, keepdim=True) / s)[:, 0]
    return (v * t0 - r + torch.log(s * h))[:, 0]


def _plain_i(v, x, deriv):
    out = torch.empty_like(x)
    near = v * v + x * x <= 3600.0
    if bool(near.any()):
        a, b = v[near], x[near]
        y = 0.25 * b * b
        term, s, ks = torch.ones_like(b), torch.ones_like(b), torch.zeros_like(b)
        for k in range(1, 121):
            term = term * (y / (k * (k + a)))
            s = s + term
            ks = ks + k * term
        if deriv:
            out[near] = (a + 2.0 * ks / s) / b
        else:
            out[near] = torch.where(a > 0, a * torch.log(0.5 * b), 0.0 * a) - torch.lgamma(a + 1.0) + torch.log(s)
    far = ~near
    if bool(far.any()):
        a, b = v[far][:, None], x[far][:, None]
        r = torch.hypot(a, b)
        h = 0.3 / torch.sqrt(r)
        th = h * torch.arange(0, 40, dtype=torch.float64, device=x.device)[None]
        th[:, 0] = 1e-300                          # the limit theta -> 0
        q = th / torch.sin(th)
        q[:, 0] = 1.0
        sh = (a / b) * q
        al, ch = torch.asinh(sh), torch.sqrt(1.0 + sh * sh)
        al0 = al[:, :1]
        e = b * (ch * torch.cos(th) - ch[:, :1]) - a * (al - al0)
        w = torch.exp(e)
        w[:, 0] *= 0.5
        s = w.sum(1, keepdim=True)
        if deriv:
            slope = (a / b) * (torch.sin(th) - th * torch.cos(th)) / torch.sin(th) ** 2 / ch
            slope[:, 0] = 0.0
            out[far] = ((w * (ch * torch.cos(th) + sh * torch.sin(th) * slope)).sum(1, keepdim=True) / s)[:, 0]
        else:
            out[far] = (r - a * al0 + torch.log(s * h / math.pi))[:, 0]
    return out


def _plain(kind, v, x, deriv=False):
    v, x = v.double(), x.double()
    out = torch.empty_like(x)
    step = 1 << 18
    for i in range(0, x.numel(), step):
        c = x[i:i + step]
        vc = v[i:i + step] if v.numel() == x.numel() else v.expand(c.numel())
        out[i:i + step] = (_plain_i if kind == "i" else _plain_k)(vc, c, deriv)
    return out


def exact(case, seed):
    op = case["op"]
    if case["n"] > 24000000:
        return None                                # over 20 seconds
    if op == "served":
        got = {torch.float64: [], torch.float32: []}
        for kind, v, x in _inputs(case, seed):
            got[x.dtype].append(_plain(kind, v, x))
        return [torch.cat(got[dt] or [torch.empty(0, dtype=torch.float64, device="cuda")])
                for dt in (torch.float64, torch.float32)]
    v, x = _inputs(case, seed)
    if op == "vmf":
        d = case["v"]
        nu = torch.tensor([0.5 * d - 1.0], dtype=torch.float64, device="cuda")
        return (nu * torch.log(x) - 0.5 * d * math.log(2.0 * math.pi) - _plain("i", nu, x),
                nu / x - _plain("i", nu, x, True))
    kind = "i" if "_i" in op else "k"
    if op.startswith("grad"):
        g = prepare(case, seed)["g"]
        return _plain(kind, v, x), g * _plain(kind, v, x, True)
    return _plain(kind, v, x, op.endswith("dx"))
