"""Performance cases: the calls that a user of the package makes, over the sizes it is used at.

A case is a dict of plain values.  ``prepare`` makes its recording and its evaluation point from a seed, ``run`` is
one pass through the public API, ``exact`` the same quantities in FP64 with plain torch, ``work`` the bytes and
operations that a pass cannot do without.

Recordings.  Rates are a few Hz, log-normal over the neurons; weights are those of the balanced network (80:20
excitatory : inhibitory, connection probability 0.1, inhibition four times as strong, a refractory self weight) plus
the estimation noise of an unfinished fit.  Evaluations only need trains of the right density, so those are drawn
bin by bin on the GPU; the recordings that are fitted are simulated from the model itself.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1502_04993_gb300 as glm
from paper_1502_04993_gb300.autograd import glm_loglik

DEV = "cuda:0"
DT = 0.001


def listed():
    return [
        # one evaluation of the smallest configuration (50 neurons, 20 s at 1 ms): launches and latency count
        dict(name="eval_n50", kind="eval", form="f16x1", n=50, bins=20_000, rate=5.0, tau=0.010),
        # the plain FP32 fit of that configuration, to the default stopping rule: hundreds of such evaluations
        dict(name="fit_f32_n50", kind="fit", form="f32", n=50, bins=20_000, rate=5.0, tau=0.010, eta=1e-10),
        # a fit of a few hundred neurons over a minute in the default form
        dict(name="fit_n203", kind="fit", form="f16x1", n=203, bins=60_001, rate=8.0, tau=0.010, eta=1e-9),
        # differentiable log-likelihood and its backward pass, in the library's default form (BF16, X split),
        # ragged sizes
        dict(name="autograd_n317", kind="autograd", form="bf16", n=317, bins=100_003, rate=8.0, tau=0.010),
        # one optimiser evaluation at paper scale: 1000 neurons, 1800 s
        dict(name="eval_n1000_t1800s", kind="eval", form="f16x1", n=1000, bins=1_800_000, rate=8.0, tau=0.010),
        # a point of a scan over the time constant: caches rebuilt for a new tau, then an evaluation
        dict(name="tau_point_n1000", kind="tau_point", form="f16x1", n=1000, bins=600_000, rate=8.0, tau=0.012),
        # two consecutive windows of a recording from host memory, each set as the problem and evaluated
        dict(name="windows_n400", kind="windows", form="f16x1", n=400, bins=200_000, rate=8.0, tau=0.010),
        # the plain FP32 form, with which fits are finished and results are checked
        dict(name="eval_f32_n300", kind="eval", form="f32", n=300, bins=60_000, rate=8.0, tau=0.010),
        # spike times off the grid: exact column integrals
        dict(name="ct_n300", kind="ct", form="bf16", n=300, seconds=30.0, rate=8.0, tau=0.010, delay=0.0015),
        # the same with the derivative in the time constant, through autograd
        dict(name="ct_tau_n600", kind="ct_tau", form="bf16", n=600, seconds=30.0, rate=8.0, tau=0.010, delay=0.001),
        # 2000 neurons with X recomputed in chunks, gradients in W, b and tau
        dict(name="chunked_tau_n2000", kind="chunked_tau", form="f16x1", n=2000, bins=524_300, chunk=262_144, rate=6.0,
             tau=0.010),
        # the filtered trains of part of a recording, for a caller's own analysis
        dict(name="filter_n1000", kind="filter", form="f16x1", n=1000, bins=400_000, t0=100_003, length=200_001,
             rate=8.0, tau=0.010, dtype="f32"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval_f32", "fit", "autograd", "tau_point", "windows", "ct", "ct_tau",
                       "chunked_tau", "filter"])
    rate = round(rng.uniform(3.0, 12.0), 2)
    tau = rng.choice([0.008, 0.010, 0.014, 0.020])
    c = dict(kind=kind, rate=rate, tau=tau)
    if kind == "eval":
        n = _log_uniform(rng, 20, 1000)
        c.update(form="f16x1", n=n, bins=_log_uniform(rng, 4_000, min(1_800_000, 1_500_000_000_000 // (n * n))))
    elif kind == "eval_f32":
        c.update(kind="eval", form="f32", n=_log_uniform(rng, 20, 500), bins=_log_uniform(rng, 4_000, 100_000))
    elif kind == "fit":
        c.update(form=rng.choice(["f32", "f16x1"]), n=_log_uniform(rng, 20, 200), bins=_log_uniform(rng, 8_000, 50_000),
                 eta=rng.choice([1e-9, 1e-10]))
    elif kind == "autograd":
        c.update(form=rng.choice(["bf16", "f16"]), n=_log_uniform(rng, 30, 900), bins=_log_uniform(rng, 10_000, 200_000))
    elif kind == "tau_point":
        c.update(form=rng.choice(["f16x1", "bf16"]), n=_log_uniform(rng, 100, 1000),
                 bins=_log_uniform(rng, 20_000, 500_000))
    elif kind == "windows":
        c.update(form="f16x1", n=_log_uniform(rng, 60, 600), bins=_log_uniform(rng, 20_000, 200_000))
    elif kind in ("ct", "ct_tau"):
        c.update(form=rng.choice(["bf16", "f16"]), n=_log_uniform(rng, 40, 700), seconds=round(rng.uniform(4.0, 30.0), 3),
                 delay=rng.choice([0.0, 0.001, 0.0015]))
    elif kind == "chunked_tau":
        bins = _log_uniform(rng, 60_000, 400_000)
        c.update(form=rng.choice(["f16x1", "bf16"]), n=_log_uniform(rng, 150, 1600), bins=bins,
                 chunk=bins // rng.randint(2, 4))
    else:
        bins = _log_uniform(rng, 20_000, 400_000)
        t0 = rng.randrange(bins // 2)
        c.update(form="f16x1", n=_log_uniform(rng, 50, 1000), bins=bins, t0=t0, length=rng.randint(1_000, bins - t0),
                 dtype=rng.choice(["f32", "f32", "bf16", "f16"]))
    return c


# ---- inputs ----


def _generator(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def _rates(case, seed):
    """Rates in Hz, log-normal around the case's rate."""
    z = torch.randn(case["n"], generator=_generator(seed, 1), device=DEV, dtype=torch.float64)
    return (case["rate"] * torch.exp(0.4 * z - 0.08)).clamp(0.3, 60.0)


def _weights(case, seed, noise=True):
    """Weights (FP64 holding FP32 values): W[i, j] is the weight of j -> i."""
    n = case["n"]
    we = 0.5 if n < 100 else 0.3 if n < 500 else 0.2
    g = _generator(seed, 2)
    W = (torch.rand((n, n), generator=g, device=DEV) < 0.1).to(torch.float64)
    W[:, : (4 * n) // 5] *= we
    W[:, (4 * n) // 5:] *= -4.0 * we
    W.fill_diagonal_(-6.25)
    if noise:
        W += 0.05 * torch.randn((n, n), generator=g, device=DEV, dtype=torch.float64)
    return W.to(torch.float32).to(torch.float64)


def _bias(case, seed):
    z = torch.randn(case["n"], generator=_generator(seed, 3), device=DEV, dtype=torch.float64)
    return (torch.log(_rates(case, seed)) + 0.1 * z).to(torch.float32).to(torch.float64)


def _trains(case, seed, bins, salt=10):
    """(rows, bins) of the spikes of independent trains, sorted by row and bin, on the GPU."""
    n, g = case["n"], _generator(seed, salt)
    p = (_rates(case, seed) * DT).to(torch.float32)
    step = max(1, (1 << 27) // bins)
    rows, at = [], []
    for r0 in range(0, n, step):
        r1 = min(n, r0 + step)
        idx = (torch.rand((r1 - r0, bins), generator=g, device=DEV) < p[r0:r1, None]).nonzero()
        rows.append(idx[:, 0] + r0)
        at.append(idx[:, 1])
    return torch.cat(rows), torch.cat(at)


def _csr(n, rows, values, dtype):
    """Host CSR arrays of spikes sorted by row."""
    offs = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(torch.bincount(rows, minlength=n).cpu().numpy(), out=offs[1:])
    return offs, values.to(dtype).cpu().numpy()


def _simulated(case, seed):
    """Host CSR of a recording simulated from the model (the fits need connections to find)."""
    n, T, a = case["n"], case["bins"], math.exp(-DT / case["tau"])
    W = _weights(case, seed, noise=False).cpu().numpy()
    rng = np.random.default_rng(int(seed) + 77)
    base = np.full(n, case["rate"] * DT)
    v, hits = np.zeros(n), []
    for t0 in range(0, T, 4096):
        u = rng.random((min(4096, T - t0), n))
        for k in range(u.shape[0]):
            s = np.flatnonzero(u[k] < np.minimum(base * np.exp(v), 0.2))
            v *= a
            if s.size:
                v += W[:, s].sum(axis=1)
                hits.append(s.astype(np.int64) * T + (t0 + k))
    key = np.sort(np.concatenate(hits))
    offs = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // T, minlength=n), out=offs[1:])
    return offs, (key % T).astype(np.int32)


def _context(case):
    """A context in the case's form, and the precision to set its problems with."""
    ctx = glm.GLM(0)
    ctx.set_x_split(case["form"] != "f16x1")
    if case["kind"] == "chunked_tau":
        ctx.set_chunk_bins(case["chunk"])
    return ctx, {"f16x1": "f16"}.get(case["form"], case["form"])


def _event_times(case, seed):
    """(rows, times) of spikes off the grid: each uniformly inside its bin."""
    rows, at = _trains(case, seed, int(case["seconds"] / DT))
    u = torch.rand(at.shape, generator=_generator(seed, 4), device=DEV, dtype=torch.float64)
    return rows, (at.to(torch.float64) + u) * DT


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    ctx, prec = _context(case)
    st = dict(case=case, ctx=ctx, prec=prec)
    if kind == "fit":
        offs, bins = _simulated(case, seed)
        ctx.set_problem(offs, bins, case["bins"], DT, case["tau"], prec=prec)
        return st
    if kind == "windows":
        st["windows"] = [_csr(n, *_trains(case, seed, case["bins"], salt), torch.int32) for salt in (10, 11)]
    elif kind in ("ct", "ct_tau"):
        offs, times = _csr(n, *_event_times(case, seed), torch.float64)
        ctx.set_problem_ct(offs, times, 0.0, case["seconds"], case["tau"], case["delay"], prec=prec)
    else:
        offs, bins = _csr(n, *_trains(case, seed, case["bins"]), torch.int32)
        ctx.set_problem(offs, bins, case["bins"], DT, case["tau"], prec=prec)
    if kind != "filter":
        st["W"] = _weights(case, seed).to(torch.float32)
        st["b"] = _bias(case, seed).to(torch.float32)
    if kind in ("autograd", "ct_tau", "chunked_tau"):
        st["W"].requires_grad_()
        st["b"].requires_grad_()
        st["tau"] = torch.tensor(case["tau"], dtype=torch.float64, requires_grad=kind != "autograd")
    return st


# ---- one pass ----


def _evaluate(ctx, W, b):
    r = ctx.loglik_grad(W, b)
    return {k: r[k] for k in ("L_rows", "L_total", "G", "gb")}


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind in ("eval", "ct"):
        return _evaluate(ctx, st["W"], st["b"])
    if kind == "fit":
        r = ctx.fit(eta=case["eta"])
        return {"W": r["W"], "b": r["b"], "L": r["report"]["L"]}
    if kind in ("autograd", "ct_tau", "chunked_tau"):
        L = glm_loglik(ctx, st["W"], st["b"], st["tau"])
        wrt = {"gW": st["W"], "gb": st["b"]}
        if st["tau"].requires_grad:
            wrt["gtau"] = st["tau"]
        return {"L": L.detach(), **dict(zip(wrt, torch.autograd.grad(L, tuple(wrt.values()))))}
    if kind == "tau_point":
        ctx.prepare(case["tau"])
        return _evaluate(ctx, st["W"], st["b"])
    if kind == "windows":
        out = []
        for offs, bins in st["windows"]:
            ctx.set_problem(offs, bins, case["bins"], DT, case["tau"], prec=st["prec"])
            out.append(_evaluate(ctx, st["W"], st["b"]))
        return out
    return {"X": ctx.filter(case["t0"], case["length"], dtype=case["dtype"])}


def work(case):
    """Bytes: the trains X (or the spikes, where the pass starts from them) and the parameters read once, the
    results written once.  Operations: two products of 2 n^2 per bin (U = W X and the gradient)."""
    n, kind = case["n"], case["kind"]
    nn, x = float(n) * n, 4.0 if case["form"] == "f32" else 2.0
    if kind in ("ct", "ct_tau"):
        cols = 2.0 * n * case["rate"] * case["seconds"]  # an arrival and a spike column per spike
        # the split trains; dL/dtau needs no third product (W dv/dtau follows from W v by a recursion)
        return {"bytes": 4.0 * n * cols + 12.0 * nn, "flops": 4.0 * nn * cols}
    spikes = 4.0 * n * case["bins"] * case["rate"] * DT
    if kind == "filter":
        out = (4.0 if case["dtype"] == "f32" else 2.0) * n * case["length"]
        return {"bytes": out + spikes * case["length"] / case["bins"], "flops": 2.0 * n * case["length"]}
    nt = float(n) * case["bins"]
    one = {"bytes": x * nt + 12.0 * nn, "flops": 4.0 * n * nt}
    if case["form"] in ("bf16", "f16"):
        one["bytes"] += x * nt  # the second part of the split X
    if kind == "fit":  # the shortest fits take a few dozen evaluations
        return {"bytes": 30.0 * one["bytes"], "flops": 30.0 * one["flops"]}
    if kind == "chunked_tau":  # from the spikes
        return {"bytes": spikes + 12.0 * nn, "flops": one["flops"]}
    if kind == "tau_point":  # the spike term is a sum over the spikes
        return {"bytes": spikes + 20.0 * nn, "flops": one["flops"] + 2.0 * n * spikes / 4.0}
    if kind == "windows":
        return {"bytes": 2.0 * (spikes + 20.0 * nn), "flops": 2.0 * (one["flops"] + 2.0 * n * spikes / 4.0)}
    return one


# ---- the same quantities in FP64 ----


class _Recursion:
    """x[t] = a x[t-1] + s[t-1] over consecutive chunks of bins (FP64): blocks of 256 bins by a triangular
    product, the carries from block to block in order."""

    B = 256

    def __init__(self, n, a):
        self.a, self.x = a, torch.zeros(n, dtype=torch.float64, device=DEV)
        m = torch.arange(self.B, device=DEV, dtype=torch.float64)
        e = m[None, :] - 1 - m[:, None]
        self.local = torch.where(e >= 0, a ** e.clamp(min=0), torch.zeros_like(e))  # [k, m]: s[k] in x[m]
        self.last = a ** (self.B - 1 - m)
        self.pw = a ** m

    def __call__(self, s):
        n, T = s.shape
        nb = -(-T // self.B)
        sp = torch.nn.functional.pad(s, (0, nb * self.B - T)).reshape(n, nb, self.B)
        ends, carry = sp @ self.last, torch.empty((n, nb), dtype=torch.float64, device=DEV)
        for k in range(nb):
            carry[:, k] = self.x
            self.x = self.x * self.a ** self.B + ends[:, k]
        return (sp @ self.local + carry[:, :, None] * self.pw).reshape(n, nb * self.B)[:, :T]


def _grid_exact(case, rows, at, W, b, want_tau=False):
    n, T, tau = case["n"], case["bins"], case["tau"]
    a = math.exp(-DT / tau)
    f, fz = _Recursion(n, a), _Recursion(n, a)
    L = torch.zeros(n, dtype=torch.float64, device=DEV)
    gb, r_z = torch.zeros_like(L), torch.zeros_like(L)
    G = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    step = max(256, ((1 << 26) // n) // 256 * 256)
    for t0 in range(0, T, step):  # whole blocks but for the last chunk
        t1 = min(T, t0 + step)
        S = torch.zeros((n, t1 - t0), dtype=torch.float64, device=DEV)
        m = (at >= t0) & (at < t1)
        S[rows[m], at[m] - t0] = 1.0
        X = f(S)
        V = W @ X
        R = torch.exp(V + b[:, None]) * DT
        L += (S * (V + b[:, None]) - R).sum(1)
        R = S - R
        gb += R.sum(1)
        G += R @ X.T
        if want_tau:
            r_z += (R * fz(V)).sum(1)
    return L, G, gb, float(r_z.sum()) * a * DT / (tau * tau)


def _ct_exact(case, rows, times, W, b):
    """Event columns (Eq. 8-14); the integral over each column by 16-node Gauss-Legendre quadrature in time."""
    n, tau, end = case["n"], case["tau"], case["seconds"]
    arr = times + case["delay"]
    arows, arr = rows[arr < end], arr[arr < end]
    cols = torch.unique(torch.cat([torch.zeros(1, dtype=torch.float64, device=DEV), arr, times]))
    length = torch.diff(cols, append=torch.full((1,), end, dtype=torch.float64, device=DEV))
    at_arr, at_spk = torch.searchsorted(cols, arr), torch.searchsorted(cols, times)
    xs, ws = np.polynomial.legendre.leggauss(16)
    L = torch.zeros(n, dtype=torch.float64, device=DEV)
    gb, G = torch.zeros_like(L), torch.zeros((n, n), dtype=torch.float64, device=DEV)
    v0, y0, gtau, eb = torch.zeros_like(L), torch.zeros_like(L), 0.0, torch.exp(b)[:, None]
    cuts = torch.searchsorted(cols, torch.arange(0.0, end, 20 * tau, dtype=torch.float64, device=DEV)).tolist()
    cuts.append(cols.numel())
    for m0, m1 in zip(cuts, cuts[1:]):
        if m0 == m1:
            continue
        c0 = cols[m0]  # the state at the block's first column starts the block
        if m0 > 0:
            h = c0 - cols[m0 - 1]
            y0, v0 = torch.exp(-h / tau) * (y0 + h * v0), torch.exp(-h / tau) * v0
        k = (at_arr >= m0) & (at_arr < m1)
        grown = torch.exp((arr[k] - c0) / tau)
        A = torch.zeros((n, m1 - m0), dtype=torch.float64, device=DEV)
        A.index_put_((arows[k], at_arr[k] - m0), grown, accumulate=True)
        A1 = torch.zeros_like(A)
        A1.index_put_((arows[k], at_arr[k] - m0), grown * (arr[k] - c0), accumulate=True)
        h, D = cols[m0:m1] - c0, length[m0:m1]
        A, A1 = A.cumsum(1) + v0[:, None], A1.cumsum(1) - y0[:, None]
        decay = torch.exp(-h / tau)
        v, y = decay * A, decay * (h * A - A1)
        v0, y0 = v[:, -1].clone(), y[:, -1].clone()
        u, z = W @ v, W @ y
        F, Gm, Ft = torch.zeros_like(u), torch.zeros_like(u), torch.zeros_like(u)
        for x, w in zip(xs, ws):
            s = 0.5 * (x + 1.0) * D
            r = torch.exp(-s / tau)
            e = torch.exp(u * r) * (0.5 * w * D)
            F += e
            Gm += e * r
            Ft += e * u * (r * s / (tau * tau))
        S = torch.zeros_like(u)
        k = (at_spk >= m0) & (at_spk < m1)
        S.index_put_((rows[k], at_spk[k] - m0), torch.ones_like(times[k]), accumulate=True)
        L += (S * (u + b[:, None]) - eb * F).sum(1)
        gb += (S - eb * F).sum(1)
        R = S - eb * Gm
        G += R @ v.T
        gtau += float((R * z).sum()) / (tau * tau) - float((eb * Ft).sum())
    return L, G, gb, gtau


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "fit":
        return None  # where a fit stops is not fixed beyond its stopping rule
    if kind == "filter":
        rows, at = _trains(case, seed, case["bins"])
        f, t0, t1 = _Recursion(n, math.exp(-DT / case["tau"])), case["t0"], case["t0"] + case["length"]
        out, step = [], 65_536
        for s0 in range(0, t1, step):
            S = torch.zeros((n, step), dtype=torch.float64, device=DEV)
            m = (at >= s0) & (at < s0 + step)
            S[rows[m], at[m] - s0] = 1.0
            X = f(S)
            if s0 + step > t0:
                out.append(X[:, max(t0 - s0, 0): t1 - s0])
        return {"X": torch.cat(out, 1)}
    W, b = _weights(case, seed), _bias(case, seed)
    if kind == "windows":
        got = [_grid_exact(case, *_trains(case, seed, case["bins"], salt), W, b) for salt in (10, 11)]
        return [{"L_rows": L, "L_total": float(L.sum()), "G": G, "gb": gb} for L, G, gb, _ in got]
    if kind in ("ct", "ct_tau"):
        L, G, gb, gtau = _ct_exact(case, *_event_times(case, seed), W, b)
    else:
        L, G, gb, gtau = _grid_exact(case, *_trains(case, seed, case["bins"]), W, b, kind == "chunked_tau")
    if kind in ("eval", "ct", "tau_point"):
        return {"L_rows": L, "L_total": float(L.sum()), "G": G, "gb": gb}
    out = {"L": L.sum(), "gW": G, "gb": gb}
    if kind != "autograd":
        out["gtau"] = torch.tensor(gtau, dtype=torch.float64)
    return out
