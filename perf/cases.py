"""What the framework's users have it compute, as measurable cases.

A case is one call a program makes through the Python binding: a solve
(``Hamiltonian.estimate``), a solve of the total model and of its bare bath with H*
formed from both, a batch of uneven solves, or a burst of requests to the serving loop.
Sizes are those of this repository's workloads, tests and benchmark. A case fixes sizes,
precision and options; the seed draws the couplings and the bath vectors.

The float64 path's results are handed on as float64. A float32 solve keeps its Krylov
vectors, its matrix products and psi = Q c in float32 and its results are good to that
precision, so they are handed on as float32.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import workloads as W
from paper_2204_08147_gb300 import rdm

_STATE: dict = {}  # the process's context and its serving context


def _context():
    """One library context per process, as a program that solves many models keeps it."""
    if "ctx" not in _STATE:
        _STATE["ctx"] = rdm.Context(0)
    return _STATE["ctx"]


def _server():
    """A second context that runs the serving loop (4 workers, 32 GiB)."""
    if "server" not in _STATE:
        ctx = rdm.Context(0)
        ctx.serve_start(32 << 30, 4)
        _STATE["server"] = ctx
    return _STATE["server"]


# ---------------------------------------------------------------- the cases

def _solve(name, model, n, n_sys, n_v, k, n_beta, lo, hi, precision="fp32", dist="gauss", alpha=0.0,
           passes="auto", recurrence="block", budget_mb=0, kind="estimate"):
    return dict(name=name, kind=kind, model=model, n=n, n_sys=n_sys, n_v=n_v, k=k, n_beta=n_beta, beta_lo=lo,
                beta_hi=hi, precision=precision, dist=dist, alpha=alpha, passes=passes, recurrence=recurrence,
                budget_mb=budget_mb)


def listed():
    return [
        # the smallest solve, where launches and host steps count: the periodic XXZ chain
        # of 10 spins in float64
        _solve("chain10_fp64", "chain", 10, 1, 16, 40, 3, 0.5, 2.0, precision="fp64", dist="rademacher"),
        # one request of the serving mix on its own: a small long-range Ising model on a
        # temperature grid
        _solve("tfim12_request", "tfim", 12, 2, 16, 45, 24, 0.1, 10.0, dist="rademacher", alpha=1.5),
        # the solvable chain experiment: rho* and ln Z_t of the chain, ln Z_b of its bath
        # (one-column blocks), H* with its constant on 12 temperatures
        _solve("chain18_hstar", "open_xy", 18, 2, 100, 30, 12, 0.1, 10.0, kind="hstar"),
        # the spin ladder, numbered leg by leg (the library reorders the bath)
        _solve("ladder20", "ladder", 20, 2, 50, 30, 16, 0.1, 10.0),
        # one field value of the entropy phase plot: many bath vectors of a small model
        _solve("sweep16_lrxy", "lrxy", 16, 2, 400, 60, 8, 0.5, 4.0, alpha=1.0),
        # the benchmark's solve
        _solve("tfim22", "tfim", 22, 2, 32, 60, 1, 1.0, 1.0, alpha=1.5),
        # long-range XXZ on a temperature grid, a quarter of the bath vectors and an eighth
        # of the states of the 25-spin configuration
        _solve("xxz22_grid", "xxz", 22, 1, 16, 40, 32, 0.1, 10.0, dist="rademacher", alpha=1.0),
        # the 30-spin configuration's shape (few bath vectors, one temperature, a block of
        # one slice) at 24 spins
        _solve("xxz24_few_vectors", "xxz", 24, 1, 4, 50, 1, 2.0, 2.0, dist="rademacher", alpha=1.5),
        # a solve held to a memory budget that its Krylov basis does not fit, odd counts
        _solve("xxz19_budget", "xxz", 19, 1, 45, 37, 20, 0.1, 10.0, dist="rademacher", alpha=1.5, budget_mb=2048),
        # the float64 path at a middle size
        _solve("tfim19_fp64", "tfim", 19, 2, 8, 60, 1, 1.0, 1.0, precision="fp64", alpha=1.5),
        # uneven small solves handed over together
        dict(name="batch48", kind="batch", requests=48, stream=20220422, n_min=8, n_max=14),
        # a burst of requests to the serving loop
        dict(name="serve24", kind="serve", requests=24, stream=20220419, n_min=12, n_max=16),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    most = max(_cost(c) for c in listed() if c["kind"] in ("estimate", "hstar"))
    while True:
        kind = rng.choice(["small", "small", "chain", "ladder", "tfim", "xxz", "xxz", "few", "budget", "fp64",
                           "hstar", "batch", "serve"])
        if kind == "batch":
            return dict(kind="batch", requests=_loguniform(rng, 3, 48), stream=rng.randrange(1 << 30), n_min=8,
                        n_max=rng.randint(10, 14))
        if kind == "serve":
            return dict(kind="serve", requests=_loguniform(rng, 2, 24), stream=rng.randrange(1 << 30), n_min=12,
                        n_max=rng.randint(13, 16))
        n_sys = rng.randint(1, 2)
        n_v = _loguniform(rng, 1, 64)
        k = rng.randint(20, 100)
        n_beta = _loguniform(rng, 1, 64)
        dist = rng.choice(["gauss", "rademacher"])
        alpha = rng.choice([1.0, 1.5])
        hi = rng.choice([1.0, 2.0, 4.0, 10.0])
        lo = hi if n_beta == 1 else 0.1
        model = rng.choice(["tfim", "xxz", "chain"])
        if kind == "small":
            c = _solve("", model, rng.randint(8, 15), n_sys, n_v, k, n_beta, lo, hi, dist=dist, alpha=alpha,
                       recurrence=rng.choice(["block", "block", "block", "single"]))
        elif kind == "chain":
            c = _solve("", "chain", rng.randint(16, 22), n_sys, n_v, k, n_beta, lo, hi, dist=dist)
        elif kind == "ladder":
            c = _solve("", "ladder", 2 * rng.randint(6, 11), 2, n_v, k, n_beta, lo, hi, dist=dist)
        elif kind == "tfim":
            c = _solve("", "tfim", rng.randint(16, 22), n_sys, n_v, k, n_beta, lo, hi, dist=dist, alpha=alpha)
        elif kind == "xxz":
            c = _solve("", rng.choice(["xxz", "lrxy"]), rng.randint(14, 22), n_sys, _loguniform(rng, 4, 400), k,
                       n_beta, lo, hi, dist=dist, alpha=alpha)
        elif kind == "few":
            c = _solve("", model, rng.randint(21, 24), 1, rng.randint(1, 4), k, 1, hi, hi, dist=dist, alpha=alpha)
        elif kind == "budget":
            c = _solve("", model, rng.randint(16, 20), n_sys, rng.randint(20, 64), k, n_beta, lo, hi, dist=dist,
                       alpha=alpha, budget_mb=2048, passes=rng.choice(["auto", "recompute"]))
        elif kind == "fp64":
            c = _solve("", model, rng.randint(8, 19), n_sys, n_v, k, min(n_beta, 16), lo, hi, precision="fp64",
                       dist=dist, alpha=alpha)
        else:
            c = _solve("", "open_xy", rng.randint(12, 20), rng.randint(1, 2), n_v, k, n_beta, lo, hi, dist=dist,
                       kind="hstar")
        if _cost(c) <= most and _basis_bytes(c) < 100e9:
            del c["name"]
            return c


def _basis_bytes(c):
    elem = 8 if c["precision"] == "fp64" else 4
    return (1 << (c["n"] + c["n_sys"])) * c["n_v"] * elem * (c["k"] + 1)


def _active_flips(c):
    """Off-diagonal products a row of H takes part in, on average."""
    n = c["n"]
    return {"chain": n / 2, "open_xy": (n - 1) / 2, "ladder": (3 * n / 2 - 2) / 2, "tfim": n}.get(
        c["model"], n * (n - 1) / 4)


def _flops(c):
    cols = (1 << c["n_sys"]) * c["n_v"]
    ds = 1 << c["n_sys"]
    per_step = 2 * _active_flips(c) + 2 + 10 * ds
    return (1 << c["n"]) * cols * c["k"] * (per_step + 2 * ds * c["n_beta"])


def _cost(c):
    """Grows as a case's time does: the products of its steps, float64 counted dearer."""
    return _flops(c) * (16 if c["precision"] == "fp64" else 1)


def work(case):
    """Bytes: each Lanczos step reads two blocks and writes one, and the whole basis is
    read once for the function's columns. Flops: the products of H with the block, the
    d_s x d_s mixings and inner products of a step, the columns at each temperature."""
    if case["kind"] in ("batch", "serve"):
        parts = [work(c) for c in _request_cases(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    elem = 8 if case["precision"] == "fp64" else 4
    block = (1 << (case["n"] + case["n_sys"])) * case["n_v"] * elem
    w = {"bytes": 4.0 * case["k"] * block, "flops": float(_flops(case))}
    if case["kind"] == "hstar":  # and the bare bath, one column per bath vector
        bath = dict(case, kind="estimate", n=case["n"] - case["n_sys"], n_sys=0)
        b = work(bath)
        w = {"bytes": w["bytes"] + b["bytes"], "flops": w["flops"] + b["flops"]}
    return w


# ---------------------------------------------------------------- inputs and one pass

def _model(c, rng):
    """The case's model with couplings drawn from rng."""
    n, ns, lam = c["n"], c["n_sys"], rng.uniform(0.5, 1.5)
    h, g, delta = rng.uniform(0.05, 0.5), rng.uniform(0.2, 2.0), rng.uniform(0.2, 1.5)
    if c["model"] == "chain":
        return W.xxz_chain(n, ns, 1.0, delta, h, lam, periodic=True)
    if c["model"] == "open_xy":
        return W.xy_open_chain(n, ns, 1.0, h)
    if c["model"] == "ladder":
        return W.spin_ladder(n // 2, min(2, n // 2 - 1), h=0.5 + g, lam=lam, numbering="leg")
    if c["model"] == "tfim":
        return W.long_range_tfim(n, ns, c["alpha"], g, lam)
    return W.long_range_xxz(n, ns, c["alpha"], delta if c["model"] == "xxz" else 0.0, h, lam)


def _betas(c):
    if c["n_beta"] == 1:
        return np.array([c["beta_hi"]])
    return np.geomspace(c["beta_lo"], c["beta_hi"], c["n_beta"])


def _request_cases(case):
    """The sizes of a batch's or burst's requests, as solves (the stream fixes them)."""
    out = []
    for r in W.serving_requests(case["requests"], seed=case["stream"], n_min=case["n_min"], n_max=case["n_max"]):
        s = r["spec"]
        model = "tfim" if np.any(s.gx) else ("xxz" if np.any(np.triu(s.jx, 2)) else "chain")
        out.append(_solve("", model, s.n_sites, s.n_sys, r["n_v"], r["k"], len(r["betas"]), 0.1, 10.0,
                          dist="rademacher", alpha=1.5))
    return out


def _inputs(case, seed):
    """The models, temperatures and bath-vector seeds of one case, from the seed alone."""
    rng = random.Random(seed)
    parts = _request_cases(case) if case["kind"] in ("batch", "serve") else [case]
    return [(c, _model(c, rng), _betas(c), rng.randrange(1 << 48)) for c in parts]


def prepare(case, seed):
    parts = _inputs(case, seed)
    state = dict(case=case, parts=parts)
    if case["kind"] == "serve":
        state["ctx"] = _server()
        return state
    if case.get("budget_mb"):
        state["ctx"] = rdm.Context(0)
        state["ctx"].attach_workspace(case["budget_mb"] << 20)
    else:
        state["ctx"] = _context()
    state["hams"] = [rdm.Hamiltonian(state["ctx"], spec) for _, spec, _, _ in parts]
    if case["kind"] == "hstar":
        state["bath"] = rdm.Hamiltonian(state["ctx"], parts[0][1], part="bath")
    return state


def _numbers(out, c):
    """The results of one solve in its precision."""
    t = np.float64 if c["precision"] == "fp64" else np.float32
    return {key: np.asarray(out[key]).astype(t) for key in ("rho", "rho_quad", "lnZ", "e0")}


def run(state):
    case, parts = state["case"], state["parts"]
    if case["kind"] == "batch":
        jobs = [dict(ham=h, betas=b, n_v=c["n_v"], k=c["k"], seed=s, precision=c["precision"], dist=c["dist"])
                for h, (c, _, b, s) in zip(state["hams"], parts)]
        return _joined([_numbers(o, c) for o, (c, _, _, _) in zip(state["ctx"].estimate_batch(jobs), parts)])
    if case["kind"] == "serve":
        ctx = state["ctx"]
        tickets = [ctx.submit(spec, b, c["n_v"], c["k"], s, precision=c["precision"], dist=c["dist"])
                   for c, spec, b, s in parts]
        return _joined([_numbers(ctx.wait(t), c) for t, (c, _, _, _) in zip(tickets, parts)])
    c, _, betas, seed = parts[0]
    opts = dict(precision=c["precision"], dist=c["dist"])
    total = state["hams"][0].estimate(betas, c["n_v"], c["k"], seed, passes=c["passes"],
                                      recurrence=c["recurrence"], **opts)
    out = _numbers(total, c)
    if case["kind"] == "hstar":
        bath = state["bath"].estimate(betas, c["n_v"], c["k"], seed, **opts)
        out["lnZ_bath"] = np.asarray(bath["lnZ"]).astype(out["lnZ"].dtype)
        out["h_star"] = np.stack([rdm.mean_force_abs(total["rho"][i], b, total["lnZ"][i], bath["lnZ"][i])
                                  for i, b in enumerate(betas)]).astype(out["rho"].dtype)
    return out


def _joined(results):
    """The results of many solves, flattened one after another by kind."""
    return {key: np.concatenate([np.ravel(r[key]) for r in results]) for key in results[0]}


# ---------------------------------------------------------------- 64-bit values

def exact(case, seed):
    """The estimator's values in 64 bits: block Lanczos with full reorthogonalisation on
    the same bath vectors, exp(-beta (T - E0)) from the eigenvectors of T. (The Gram form
    and the quadrature form are one number while Q^T Q = I.) e0 is a by-product of the
    finite-precision recurrence and has no such value."""
    parts = _inputs(case, seed)
    # seconds on one GPU, roughly: the products of H, the projections on the basis, and
    # a millisecond per term and step for the launches of small models
    secs = 0.0
    for c, spec, _, _ in parts:
        elems = (1 << (c["n"] + c["n_sys"])) * c["n_v"]
        secs += c["k"] * (elems * 8 * (3 * _active_flips(c) + 4 * c["k"]) / 2e12 + 3e-5 * _active_flips(c) + 2e-3)
    if secs > 12 or (not torch.cuda.is_available() and secs > 0.2):
        return None
    results = []
    for c, spec, betas, s in parts:
        rho, lnz = _lanczos64(c, spec, betas, s)
        r = {"rho": rho, "rho_quad": rho, "lnZ": lnz, "e0": None}
        if c.get("recurrence") == "single":
            r["rho_quad"] = None  # its quadrature form has only the diagonal
        if case["kind"] == "hstar":
            _, lnz_b = _lanczos64(dict(c, n=c["n"] - c["n_sys"], n_sys=0), W.bath_spec(spec), betas, s)
            r["lnZ_bath"] = lnz_b
            r["h_star"] = np.stack([_minus_log(rho[i], b) - (lnz[i] - lnz_b[i]) / b * np.eye(rho.shape[1])
                                    for i, b in enumerate(betas)])
        results.append(r)
    if case["kind"] in ("batch", "serve"):
        out = _joined([{k: v for k, v in r.items() if v is not None} for r in results])
        out["e0"] = None
        return out
    return results[0]


def _minus_log(rho, beta):
    w, v = np.linalg.eigh(rho)
    return -(v * np.log(w)) @ v.T / beta


def _signed(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _shift(z, s):
    return (z >> s) & ((1 << (64 - s)) - 1)


def _splitmix(seed, n):
    """Output n of SplitMix64 (Steele, Lea & Flood 2014), as int64 bit patterns."""
    z = _signed(seed & (2 ** 64 - 1)) + n * _signed(0x9E3779B97F4A7C15)
    z = (z ^ _shift(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shift(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ _shift(z, 31)


def _bath_vector(dist, seed, l, d_b, dev):
    b = torch.arange(d_b, dtype=torch.int64, device=dev)
    if dist == "rademacher":
        z = _splitmix(seed, ((l << 40) | b) + 1)
        return torch.where(z < 0, -1.0, 1.0).to(torch.float64) / math.sqrt(d_b)
    u = [(_shift(_splitmix(seed, ((l << 40) | (2 * b + i)) + 1), 11).to(torch.float64) + 0.5) * 2.0 ** -53
         for i in (0, 1)]
    g = torch.sqrt(-2.0 * torch.log(u[0])) * torch.cos(2.0 * math.pi * u[1])
    return g / g.norm()


class _Operator:
    """H on the last axis (the 2^N states) of a float64 tensor, term by term on views."""

    def __init__(self, spec, dev):
        self.spec, n = spec, spec.n_sites
        s = torch.arange(1 << n, dtype=torch.int64, device=dev)
        z = [1.0 - 2.0 * ((s >> (n - 1 - q)) & 1).to(torch.float64) for q in range(n)]
        self.diag = torch.zeros(1 << n, dtype=torch.float64, device=dev)
        self.pairs = []
        self.bound = 0.0
        for a in range(n):
            self.diag += float(spec.hz[a]) * z[a]
            self.bound += abs(float(spec.hz[a])) + abs(float(spec.gx[a]))
            for b in range(a + 1, n):
                f = spec.lambda_sb if a < spec.n_sys <= b else 1.0
                jx, jy, jz = (float(f * m[a, b]) for m in (spec.jx, spec.jy, spec.jz))
                self.bound += abs(jx) + abs(jy) + abs(jz)
                if jz:
                    self.diag += jz * z[a] * z[b]
                if jx or jy:
                    self.pairs.append((a, b, jx + jy, jx - jy))

    def __call__(self, x):
        n, lead = self.spec.n_sites, x.shape[:-1]
        y = x * self.diag
        for a, b, odd, even in self.pairs:
            shape = (*lead, 1 << a, 2, 1 << (b - a - 1), 2, 1 << (n - 1 - b))
            xv, yv = x.view(shape), y.view(shape)
            for i in (0, 1):
                if odd:
                    yv[..., i, :, 1 - i, :].add_(xv[..., 1 - i, :, i, :], alpha=odd)
                if even:
                    yv[..., i, :, i, :].add_(xv[..., 1 - i, :, 1 - i, :], alpha=even)
        for a in range(n):
            if self.spec.gx[a]:
                shape = (*lead, 1 << a, 2, 1 << (n - 1 - a))
                xv, yv = x.view(shape), y.view(shape)
                for i in (0, 1):
                    yv[..., i, :].add_(xv[..., 1 - i, :], alpha=float(self.spec.gx[a]))
        return y


def _orthonormal(z, floor):
    """z = S q for each batch entry (rows): q with orthonormal or zero rows."""
    lam, v = torch.linalg.eigh(z @ z.transpose(1, 2))
    lam, v = lam.flip(1), v.flip(2)
    keep = (lam > 1e-13 * lam[:, :1]) & (lam > floor * floor)
    root = torch.where(keep, lam.clamp_min(1e-300).sqrt(), torch.ones_like(lam))
    q = (v.transpose(1, 2) @ z) * torch.where(keep, 1.0 / root, torch.zeros_like(lam))[:, :, None]
    s = v * torch.where(keep, root, torch.zeros_like(lam))[:, None, :]
    g = q @ q.transpose(1, 2)  # the identity but for rounding: one Newton step towards it
    e = torch.diag_embed(keep.to(torch.float64))
    return (1.5 * e - 0.5 * g) @ q, s @ (0.5 * (g + e))


def _lanczos64(c, spec, betas, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ds, d_b, k, n_v = spec.d_s, spec.d_b, c["k"], c["n_v"]
    single = c.get("recurrence") == "single"
    H = _Operator(spec, dev)
    chunk = max(1, min(n_v, int(30e9 // (spec.dim * ds * k * 8))))
    ts, cross = [], []
    for l0 in range(0, n_v, chunk):
        nv = min(chunk, n_v - l0)
        start = torch.zeros(nv, ds, spec.dim, dtype=torch.float64, device=dev)
        for l in range(nv):
            v = _bath_vector(c["dist"], seed, l0 + l, d_b, dev)
            for i in range(ds):
                start[l, i, i * d_b:(i + 1) * d_b] = v
        # single recurrences: every column is a recurrence of its own
        q = start.reshape(nv * ds, 1, spec.dim) if single else start
        w = q.shape[1]
        basis = torch.zeros(q.shape[0], k * w, spec.dim, dtype=torch.float64, device=dev)
        t = torch.zeros(q.shape[0], k * w, k * w, dtype=torch.float64, device=dev)
        for j in range(k):
            basis[:, j * w:(j + 1) * w] = q
            z = H(q.contiguous())
            done = basis[:, :(j + 1) * w]
            p = z @ done.transpose(1, 2)
            t[:, j * w:(j + 1) * w, j * w:(j + 1) * w] = p[:, :, j * w:]
            z = z - p @ done
            z = z - (z @ done.transpose(1, 2)) @ done
            if j + 1 < k:
                q, s = _orthonormal(z, 1e-11 * H.bound)
                t[:, (j + 1) * w:(j + 2) * w, j * w:(j + 1) * w] = s.transpose(1, 2)
                t[:, j * w:(j + 1) * w, (j + 1) * w:(j + 2) * w] = s
        ts.append(0.5 * (t + t.transpose(1, 2)).cpu())
        if single:
            cross.append((basis.view(nv, ds, k, spec.dim)).clone() if n_v * ds * k * spec.dim < 2e9 else None)
        del basis, t, q, start
    lam, v = torch.linalg.eigh(torch.cat(ts))
    e0 = float(lam.min())
    rho, lnz = [], []
    for beta in betas:
        if single:  # psi_i = Q_i f(T_i) e1 for every column, then their Gram
            f = (v * torch.exp(-0.5 * beta * (lam - e0))[:, None, :]) @ v[:, :1, :].transpose(1, 2)
            psi = torch.einsum("lik,likd->lid", f.view(n_v, ds, k).to(dev), torch.cat(cross))
            g = (psi @ psi.transpose(1, 2)).sum(0).cpu().numpy()
        else:
            f = v[:, :ds, :]
            g = ((f * torch.exp(-beta * (lam - e0))[:, None, :]) @ f.transpose(1, 2)).sum(0).numpy()
        tr = float(np.trace(g))
        rho.append(0.5 * (g + g.T) / tr)
        lnz.append(math.log(d_b * tr / n_v) - beta * e0)
    return np.stack(rho), np.array(lnz)
