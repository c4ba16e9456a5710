"""What users of this library have it do, as measurable cases.

A case is one call sequence of the public API (``Market``, ``Batch``) on a
market that a program already holds:

* ``sweep``: a block of ``k`` sweeps from the market's current potentials, then
  the potentials (the paper's timing protocol: a fixed number of iterations;
  repeated passes go on from where the last one ended);
* ``solve``: from u = v = 1 to a marginal residual, then potentials and match
  count;
* ``batch``: many independent markets solved together;
* ``topk`` / ``mu``: ranked partner lists of every user of a side, and a block
  of the matching, at potentials like those of a solved market;
* ``request``: a whole serving request: a market created from device factors,
  solved, its potentials and both sides' top-10 lists read, and released;
* ``resolve``: new factors into a resident market (host or device), then the
  warm re-solve.

Sizes, distributions, sigma and dimensions are those of this repository's
generators (``synth/markets.py``), tests and benchmark: 100 to 1e6 users per
side, d from 4 to 128, BF16 and FP32 factors, e4m3 with one scale per row or
per side, popularity biases, capacities of 1 to 5.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_19214_gb300 as tu

DEV = "cuda"

# defaults of a case (a listed or drawn case names what differs)
_BASE = dict(kind="sweep", path="fused", fmt="bf16", N=1000, M=1000, d=64, sigma=0.5, bias_x=True, bias_y=True,
             caps=1, dist="normal", k=1, stream=True, host=False, tol=1e-6, lo=0, hi=0, count=0)


def listed():
    return [
        # the smallest solve in the configurations: a balanced plain market, latency and launches
        dict(name="solve_1k_d16", kind="solve", N=1000, M=1000, d=16, sigma=1.0, bias_x=False, bias_y=False),
        # the paper's timing shape, N = M = 1e4, D = 50, a block of sweeps
        dict(name="sweep_paper_10k_d50", N=10_000, M=10_000, d=50, sigma=1.0, bias_x=False, bias_y=False,
             dist="uniform", k=10),
        # an ordinary market of the mini-batch path: popularity on both sides, ragged sizes
        dict(name="sweep_100k_d64", N=100_003, M=79_999, d=64, caps=3),
        # the headline market
        dict(name="sweep_1m_d64", N=1_000_000, M=1_000_000, d=64),
        # long factors (four 128-byte blocks per packed row)
        dict(name="sweep_d100", N=50_001, M=70_000, d=100, sigma=1.0, bias_x=False),
        # FP8 factors, one scale per row (quantized by the library)
        dict(name="sweep_fp8_rows_100k", fmt="fp8rows", N=100_000, M=80_000, d=64),
        # strong preferences: exponents beyond one shift per half-sweep
        dict(name="sweep_wide_100k", N=80_000, M=100_001, d=64, sigma=0.01),
        # the materialised-kernel path on the job market
        dict(name="dense_job_20kx10k", path="dense", fmt="fp32", N=20_000, M=10_000, d=32, bias_x=False, caps=5,
             k=10),
        # independent markets of very different sizes in one batch
        dict(name="batch_solve_56", kind="batch", count=56, lo=100, hi=50_000, d=32, sigma=1.0, bias_x=False,
             bias_y=False, caps=3),
        # recommendation lists of every user of a solved market
        dict(name="topk10_100k", kind="topk", N=100_000, M=60_000, d=64, k=10),
        # a block of the matching, at odd offsets
        dict(name="mu_block_8kx10k", kind="mu", N=10_007, M=12_001, d=50),
        # one serving request from factors to lists
        dict(name="request_20k_d32", kind="request", N=20_000, M=15_001, d=32, sigma=1.0, bias_x=False,
             bias_y=False, caps=3, stream=True),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "solve", "dense", "dense", "batch", "topk", "mu", "request",
                       "resolve"])
    bx, by = rng.random() < 0.5, rng.random() < 0.5
    c = dict(kind=kind, sigma=rng.choice([0.5, 1.0]), bias_x=bx, bias_y=by, caps=rng.choice([1, 3, 5]),
             stream=rng.random() < 0.7)
    if kind == "dense":
        c.update(kind="sweep", path="dense", fmt="fp32", N=_logint(rng, 200, 40_000), M=_logint(rng, 200, 40_000),
                 d=_logint(rng, 8, 64), k=rng.choice([1, 4, 10]))
    elif kind == "sweep":
        c.update(fmt=rng.choice(["bf16", "bf16", "bf16", "fp8rows", "fp8side"]), N=_logint(rng, 100, 400_000),
                 M=_logint(rng, 100, 400_000), d=_logint(rng, 4, 128), k=rng.choice([1, 2, 5]))
        if c["fmt"] == "bf16" and rng.random() < 0.25:
            c.update(sigma=0.01, d=_logint(rng, 32, 128))
    elif kind in ("solve", "request", "resolve"):
        c.update(N=_logint(rng, 500, 60_000), M=_logint(rng, 500, 60_000), d=rng.choice([16, 32, 50, 64]),
                 host=kind == "resolve" and rng.random() < 0.5)
    elif kind == "batch":
        c.update(count=rng.randint(8, 64), lo=100, hi=_logint(rng, 1000, 50_000), d=rng.choice([16, 32, 50]),
                 bias_x=False, bias_y=False, sigma=1.0)
    elif kind == "topk":
        c.update(N=_logint(rng, 1000, 100_000), M=_logint(rng, 1000, 100_000), d=rng.choice([16, 32, 50, 64]),
                 k=rng.choice([5, 10, 10, 20]))
    else:
        c.update(N=_logint(rng, 500, 20_000), M=_logint(rng, 500, 20_000), d=rng.choice([16, 50, 64]))
    return c


def _full(case):
    return {**_BASE, **case}


# ---------------------------------------------------------------- inputs


def _factors(g, rows, c):
    if c["dist"] == "uniform":
        x = torch.rand(rows, c["d"], generator=g, device=DEV)
    else:
        x = torch.randn(rows, c["d"], generator=g, device=DEV)
    x = x / math.sqrt(c["d"])
    return x.to(torch.bfloat16) if c["fmt"] == "bf16" else x


def _caps(rng, rows, most):
    return np.ones(rows) if most == 1 else rng.integers(1, most + 1, size=rows).astype(np.float64)


def _inputs(c, seed):
    """Factors and biases on the device, capacities on the host (as the API takes them)."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    rng = np.random.default_rng(seed)
    N, M = c["N"], c["M"]
    i = {n: _factors(g, r, c) for n, r in (("F", N), ("K", N), ("G", M), ("L", M))}
    for n, r in (("bias_x", N), ("bias_y", M)):
        i[n] = torch.randn(r, generator=g, device=DEV).exp() if c[n] else None
    i["n"] = _caps(rng, N, 1 if c["path"] == "dense" else c["caps"])
    i["m"] = _caps(rng, M, c["caps"])
    if c["kind"] in ("topk", "mu"):
        # potentials like a solved market's: popularity cancelled, capacities and noise left
        for n, r, b in (("log_u", N, i["bias_x"]), ("log_v", M, i["bias_y"])):
            p = 0.1 * torch.randn(r, generator=g, device=DEV) - 0.5 * math.log(r)
            i[n] = p - b / (2 * c["sigma"]) if b is not None else p
    return i


def _market(c, i, stream):
    if stream is not None:  # the inputs come from the current stream
        stream.wait_stream(torch.cuda.current_stream())
    return tu.Market(i["F"], i["K"], i["G"], i["L"], i["n"], i["m"], c["sigma"], bias_x=i["bias_x"],
                     bias_y=i["bias_y"], path=c["path"], stream=stream,
                     fp8={"fp8rows": True, "fp8side": "side"}.get(c["fmt"], False))


def _batch_cases(c):
    rng = np.random.default_rng([1003, c["count"], c["hi"]])  # the sizes belong to the case
    ln = rng.uniform(math.log(c["lo"]), math.log(c["hi"]), size=(c["count"], 2))
    sizes = np.rint(np.exp(ln)).astype(int)
    return [{**c, "N": int(a), "M": int(b), "caps": c["caps"] if j % 2 else 1} for j, (a, b) in enumerate(sizes)]


def _batch_inputs(c, seed):
    """Every market's inputs, its factors slices of one pool per matrix."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    rng = np.random.default_rng(seed + 1)
    pools = {n: _factors(g, c["hi"], c) for n in "FKGL"}
    out = []
    for one in _batch_cases(c):
        i = dict(bias_x=None, bias_y=None, n=_caps(rng, one["N"], one["caps"]), m=_caps(rng, one["M"], one["caps"]))
        for n, rows in (("F", one["N"]), ("K", one["N"]), ("G", one["M"]), ("L", one["M"])):
            at = int(rng.integers(0, c["hi"] - rows + 1))
            i[n] = pools[n][at:at + rows]
        out.append((one, i))
    return out


def _drift(i, c, seed):
    """The factors of a later request for the same market: N(0, 0.01^2) away."""
    g = torch.Generator(device=DEV).manual_seed(seed + 1_000_003)
    return [(i[n].float() + 0.01 * torch.randn(i[n].shape, generator=g, device=DEV)).to(i[n].dtype) for n in "FKGL"]


def prepare(case, seed):
    c = _full(case)
    stream = torch.cuda.Stream() if c["stream"] else None
    s = dict(case=c, stream=stream)
    if c["kind"] == "batch":
        s["markets"] = [_market(one, i, stream) for one, i in _batch_inputs(c, seed)]
        s["batch"] = tu.Batch(s["markets"], stream=stream)
        return s
    i = _inputs(c, seed)
    if c["kind"] == "request":
        s["inputs"] = i
        return s
    s["market"] = _market(c, i, stream)
    if c["kind"] in ("topk", "mu"):
        s["market"].set_potentials(i["log_u"], i["log_v"])
    if c["kind"] == "resolve":
        s["market"].solve(c["tol"], 2000)
        new = _drift(i, c, seed)
        s["factors"] = [x.cpu().pin_memory() for x in new] if c["host"] else new
    return s


# ---------------------------------------------------------------- one pass


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "batch":
        _, infos = state["batch"].solve(c["tol"], 2000)
        pots = [m.potentials() for m in state["markets"]]
        return dict(log_u=torch.cat([p[0] for p in pots]), log_v=torch.cat([p[1] for p in pots]),
                    matches=np.array([x["match_count"] for x in infos], np.float32))
    if kind == "request":
        m = _market(c, state["inputs"], state["stream"])
        info = m.solve(c["tol"], 2000)
        lu, lv = m.potentials()
        _, sx = m.topk(0, 10)
        _, sy = m.topk(1, 10)
        m.close()
        return dict(log_u=lu, log_v=lv, score_x=sx, score_y=sy, matches=info["match_count"])
    m = state["market"]
    if kind == "topk":
        idx, score = m.topk(0, c["k"])
        return dict(idx=idx, score=score)
    if kind == "mu":
        x0, y0 = c["N"] // 7, c["M"] // 9
        return m.mu_block(x0, c["N"] - 2 * x0 + 1, y0, c["M"] - 2 * y0 + 1)
    if kind == "sweep":
        m.sweep(c["k"])
        lu, lv = m.potentials()
        return dict(log_u=lu, log_v=lv)
    if kind == "resolve":
        m.update_factors(*state["factors"])
        info = m.solve(c["tol"], 2000, warm_start=True)
    else:
        info = m.solve(c["tol"], 2000)
    lu, lv = m.potentials()
    return dict(log_u=lu, log_v=lv, matches=info["match_count"])


# ---------------------------------------------------------------- work


_SOLVE_SWEEPS = 4  # sweeps that a solve needs (with its certificate about half a sweep more)


def work(case):
    """Packed factors, biases, capacities and FP64 potentials read once, results
    written once; a materialised kernel matrix is read once per sweep (it exceeds
    what the chip holds, and a sweep needs the one before). flops: the inner
    products, twice per sweep and once per list or block."""
    c = _full(case)
    ones = _batch_cases(c) if c["kind"] == "batch" else [c]
    size = {"bf16": 2, "fp32": 4}.get(c["fmt"], 1)
    total = dict(bytes=0.0, flops=0.0)
    for one in ones:
        N, M, d = one["N"], one["M"], one["d"]
        pairs, side = float(N) * M, N + M
        factors, state, result = side * 2 * d * size, side * (8 + 8 + 4), side * 4
        if c["kind"] == "topk":
            b, f = factors + side * 8 + N * c["k"] * 8, pairs * 4 * d
        elif c["kind"] == "mu":
            nx, ny = N - 2 * (N // 7) + 1, M - 2 * (M // 9) + 1
            b, f = (nx + ny) * (2 * d * size + 8) + 4.0 * nx * ny, 4.0 * d * nx * ny
        elif c["kind"] == "sweep" and c["path"] == "dense":
            b, f = c["k"] * (4 * pairs + state) + result, 4.0 * pairs * c["k"]
        else:
            k = c["k"] if c["kind"] == "sweep" else _SOLVE_SWEEPS
            b, f = factors + 2 * state + result, k * 2 * pairs * 4 * d
            if c["kind"] == "request":
                b, f = b + side * 80, f + 2 * pairs * 4 * d
        total["bytes"] += b
        total["flops"] += f
    return total


# ---------------------------------------------------------------- 64 bits


def _as_held(c, a, b):
    """[a | b] in float64, with the rounding that the market's format asks for."""
    x = torch.cat([a, b], 1)
    if c["fmt"] == "bf16" or c["fmt"] == "fp32":
        return x.double()
    mx = x.abs().amax(1, keepdim=True) if c["fmt"] == "fp8rows" else x.abs().amax().reshape(1, 1)
    k = torch.ceil(torch.log2(mx.double() / 448))
    k = torch.where(torch.ldexp(torch.full_like(k, 448.0), k - 1) >= mx, k - 1, k)
    k = torch.where(torch.ldexp(torch.full_like(k, 448.0), k) < mx, k + 1, k)
    sc = torch.where(mx > 0, torch.exp2(k), torch.ones_like(k))
    return (x.double() / sc).float().to(torch.float8_e4m3fn).double() * sc


def _log_sums(A, B, ell, inv2s):
    """log sum_c exp(<a_r, b_c> inv2s + ell_c) for every row of A, a slab of rows at a time."""
    out = torch.empty(A.shape[0], dtype=torch.float64, device=DEV)
    step = max(1, (1 << 27) // B.shape[0])
    for r in range(0, A.shape[0], step):
        t = torch.addmm(ell[None, :], A[r:r + step], B.T, alpha=inv2s)
        out[r:r + step] = torch.logsumexp(t, 1)
    return out


def _tau(log_p, log_o, dm):
    """Maximiser of the dual along (partner + tau, own - tau), dm = sum mass_partner - sum mass_own."""
    P, O = torch.logsumexp(2 * log_p, 0), torch.logsumexp(2 * log_o, 0)
    if dm == 0:
        return 0.25 * (O - P)
    L = math.log(abs(dm))
    q = torch.log1p(torch.sqrt(1 + torch.exp(math.log(4) + P + O - 2 * L)))
    return 0.5 * (L + q - math.log(2) - P) if dm > 0 else 0.5 * (math.log(2) + O - L - q)


def _iterate(c, i, sweeps, settle=False):
    """`sweeps` sweeps with the translation step from u = v = 1 (settle: until nothing moves)."""
    A, B = _as_held(c, i["F"], i["K"]), _as_held(c, i["G"], i["L"])
    inv2s = 0.5 / c["sigma"]
    bx, by = (i[n].double() * inv2s if i[n] is not None else 0.0 for n in ("bias_x", "bias_y"))
    n, m = (torch.from_numpy(i[x]).to(DEV) for x in ("n", "m"))
    dm = float(i["m"].sum() - i["n"].sum())
    lu, lv = torch.zeros_like(n), torch.zeros_like(m)

    def step(A, B, b_own, b_par, l_par, mass):
        log_s = math.log(0.5) + b_own + _log_sums(A, B, l_par + b_par, inv2s)
        hl = 0.5 * torch.log(mass)
        z = log_s - hl
        return hl - torch.where(z > 0, z + torch.log1p(torch.sqrt(1 + torch.exp(-2 * z))), torch.asinh(torch.exp(z)))

    for _ in range(sweeps):
        was = lu
        t = _tau(lv, lu, dm)
        lv, lu = lv + t, lu - t
        lu = step(A, B, bx, by, lv, n)
        t = _tau(lu, lv, -dm)
        lu, lv = lu + t, lv - t
        lv = step(B, A, by, bx, lu, m)
        if settle and float((lu - was).abs().max()) < 1e-12:
            break
    return lu, lv, float(i["m"].sum()) - float(torch.exp(2 * lv).sum())


def _scores(c, i, lu, lv, k, side=0):
    """The k largest log mu of every user of a side."""
    A, B = _as_held(c, i["F"], i["K"]), _as_held(c, i["G"], i["L"])
    inv2s = 0.5 / c["sigma"]
    ex, ey = (p + (i[b].double() * inv2s if i[b] is not None else 0.0) for p, b in ((lu, "bias_x"), (lv, "bias_y")))
    if side == 1:
        A, B, ex, ey = B, A, ey, ex
    out = torch.empty((A.shape[0], k), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 26) // B.shape[0])
    for r in range(0, A.shape[0], step):
        t = torch.addmm(ey[None, :], A[r:r + step], B.T, alpha=inv2s)
        out[r:r + step] = torch.topk(t, k, 1).values + ex[r:r + step, None]
    return out


def exact(case, seed):
    c = _full(case)
    if c["kind"] == "batch":
        ones = _batch_inputs(c, seed)
        if sum(float(one["N"]) * one["M"] for one, _ in ones) > 7e9:
            return None
        got = [_iterate(one, i, 7) for one, i in ones]
        return dict(log_u=torch.cat([g[0] for g in got]), log_v=torch.cat([g[1] for g in got]),
                    matches=np.array([g[2] for g in got]))
    pairs = float(c["N"]) * c["M"]
    cost = pairs * (c["d"] + 24) / 90  # about that of a pair with d = 64
    if c["kind"] == "sweep":
        if cost * c["k"] > 9e9:
            return None
        lu, lv, _ = _iterate(c, _inputs(c, seed), c["k"])
        return dict(log_u=lu, log_v=lv)
    i = _inputs(c, seed)
    if c["kind"] == "topk":
        if cost > 1e10:
            return None
        return dict(idx=None, score=_scores(c, i, i["log_u"].double(), i["log_v"].double(), c["k"]))
    if c["kind"] == "mu":
        x0, y0 = c["N"] // 7, c["M"] // 9
        rx, ry = slice(x0, x0 + c["N"] - 2 * x0 + 1), slice(y0, y0 + c["M"] - 2 * y0 + 1)
        inv2s = 0.5 / c["sigma"]
        ex, ey = (i[p].double() + (i[b].double() * inv2s if i[b] is not None else 0.0)
                  for p, b in (("log_u", "bias_x"), ("log_v", "bias_y")))
        A, B = _as_held(c, i["F"], i["K"])[rx], _as_held(c, i["G"], i["L"])[ry]
        return torch.exp(torch.addmm(ey[None, ry], A, B.T, alpha=inv2s) + ex[rx, None])
    if cost * 16 > 1.6e10:
        return None
    if c["kind"] == "resolve":
        i["F"], i["K"], i["G"], i["L"] = _drift(i, c, seed)
    lu, lv, matches = _iterate(c, i, max(16, min(400, int(1.6e10 / cost))), settle=True)
    if c["kind"] == "request":
        return dict(log_u=lu, log_v=lv, score_x=_scores(c, i, lu, lv, 10), score_y=_scores(c, i, lu, lv, 10, 1),
                    matches=matches)
    return dict(log_u=lu, log_v=lv, matches=matches)
