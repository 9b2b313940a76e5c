"""The calls that programs make of this library, sized over the range they use, for timing and comparison.

Five kinds of call:
  step     load samples, take quantiles, evaluate the grid: one whole re-optimisation
  grid     evaluate a grid on samples loaded before (FP32, FP64, EXACT or ENVELOPE)
  dual     the exact minimum over gamma >= 0 on samples loaded before
  load     load (range check and segmented sort), quantiles, the sorted samples
  noalloc  the FP32 pass that allocates nothing
A case gives a kind and its sizes; `ragged` varies the classes' sizes, supports and input lengths.
"""
import math

import numpy as np
import torch

from paper_2607_16892_gb300 import kvdro as kv

MODES = {"fp32": kv.KVDRO_FP32, "fp64": kv.KVDRO_FP64, "exact": kv.KVDRO_EXACT, "envelope": kv.KVDRO_ENVELOPE}
# Most work of a drawn case: (regime, class, r, lam, sample) terms of the per-term modes, cells of
# the others; each at or below the largest listed case of its kind.
MOST_TERMS = {"fp32": 6.7e12, "exact": 1.0e12, "fp64": 5.2e10, "envelope": 1.3e8, "dual": 8.4e6}


def listed():
    return [
        # Small service, three request classes: everything from raw samples to reservations, results
        # read by the host, once per re-optimisation; latency and launches count.
        {"name": "step_small_fp64", "kind": "step", "mode": "fp64", "K": 3, "N": 1000, "L": 8192, "R": 512, "NL": 32,
         "E": 3, "M": 1, "F": 5, "rho": 20.0, "ragged": False, "tail": False, "S": False},
        # The same grid re-evaluated on loaded samples (a knob changed): the smallest grid call.
        {"name": "grid_small_fp32", "kind": "grid", "mode": "fp32", "K": 3, "N": 1000, "L": 8192, "R": 512, "NL": 32,
         "E": 3, "M": 1, "F": 5, "rho": 20.0, "ragged": False, "tail": False, "S": False},
        # The ordinary call: eight classes with a day of samples each, a fine r and lam grid.
        {"name": "grid_k8_fp32", "kind": "grid", "mode": "fp32", "K": 8, "N": 100000, "L": 32768, "R": 4096, "NL": 128,
         "E": 8, "M": 1, "F": 5, "rho": 10.0, "ragged": False, "tail": False, "S": False},
        # The same classes where the caller wants double precision, on a coarser r grid.
        {"name": "grid_k8_fp64", "kind": "grid", "mode": "fp64", "K": 8, "N": 100000, "L": 32768, "R": 512, "NL": 128,
         "E": 8, "M": 1, "F": 5, "rho": 10.0, "ragged": False, "tail": False, "S": False},
        # Long outputs with a heavy tail (agents, reasoning): a wide support, many samples, exact mode.
        {"name": "grid_heavytail_exact", "kind": "grid", "mode": "exact", "K": 16, "N": 1000000, "L": 131072, "R": 480,
         "NL": 128, "E": 3, "M": 1, "F": 5, "rho": 10.0, "ragged": False, "tail": True, "S": False},
        # Classes as they come: unequal sizes, supports and input lengths, sizes off every tile, more
        # lam values than one block, and the S array as well.
        {"name": "grid_ragged_exact", "kind": "grid", "mode": "exact", "K": 5, "N": 40003, "L": 20011, "R": 1001,
         "NL": 200, "E": 5, "M": 3, "F": 5, "rho": 15.0, "ragged": True, "tail": False, "S": True},
        # A sweep over cost regimes (32 of a cost study), the largest per-term pass listed here.
        {"name": "sweep_fp32", "kind": "grid", "mode": "fp32", "K": 8, "N": 200000, "L": 32768, "R": 2048, "NL": 64,
         "E": 16, "M": 32, "F": 5, "rho": 1000.0, "ragged": False, "tail": False, "S": False},
        # A wider sweep in the mode that costs O(1) per cell.
        {"name": "sweep_envelope", "kind": "grid", "mode": "envelope", "K": 8, "N": 200000, "L": 32768, "R": 2048,
         "NL": 64, "E": 16, "M": 128, "F": 5, "rho": 1000.0, "ragged": False, "tail": False, "S": False},
        # The sweep without a lam grid: the exact worst case of every regime, radius, class and r.
        {"name": "sweep_dual", "kind": "dual", "mode": "dual", "K": 8, "N": 200000, "L": 32768, "R": 2048, "NL": 1,
         "E": 16, "M": 32, "F": 5, "rho": 1000.0, "ragged": False, "tail": False, "S": False},
        # The cost tables of a block-coordinate descent: every integer reservation, a radius per class.
        {"name": "dual_tables", "kind": "dual", "mode": "dual", "K": 6, "N": 300, "L": 8192, "R": 8193, "NL": 1, "E": 6,
         "M": 1, "F": 5, "rho": 10.0, "ragged": False, "tail": False, "S": False},
        # Rolling horizon: 32 classes' samples replaced, sorted and their 64 fractiles taken.
        {"name": "load_drift", "kind": "load", "mode": "load", "K": 32, "N": 1000000, "L": 32768, "R": 1, "NL": 1, "E": 1,
         "M": 1, "F": 64, "rho": 10.0, "ragged": False, "tail": False, "S": False},
        # An engine whose memory is all given to its cache: one call, nothing allocated.
        {"name": "noalloc_small", "kind": "noalloc", "mode": "fp32", "K": 4, "N": 5000, "L": 8192, "R": 512, "NL": 64,
         "E": 4, "M": 1, "F": 5, "rho": 10.0, "ragged": True, "tail": False, "S": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind, mode = rng.choice([("step", "fp32"), ("step", "fp64"), ("grid", "fp32"), ("grid", "fp32"), ("grid", "exact"),
                             ("grid", "fp64"), ("grid", "envelope"), ("dual", "dual"), ("load", "load"),
                             ("noalloc", "fp32")])
    c = {"kind": kind, "mode": mode, "K": _log_int(rng, 1, 32), "N": _log_int(rng, 300, 1000000),
         "L": _log_int(rng, 2000, 131072), "R": _log_int(rng, 100, 8192), "NL": _log_int(rng, 8, 128 if mode == "fp64" else 256),
         "E": rng.randint(1, 16), "M": 1 if rng.random() < 0.5 else _log_int(rng, 2, 128), "F": rng.randint(1, 64),
         "rho": math.exp(rng.uniform(math.log(2.0), math.log(1000.0))), "ragged": rng.random() < 0.7,
         "tail": rng.random() < 0.3, "S": False}
    if kind == "noalloc":  # its scratch holds 32 MB
        c.update(K=rng.randint(1, 6), N=_log_int(rng, 300, 100000), L=_log_int(rng, 2000, 65536), M=rng.randint(1, 4),
                 R=_log_int(rng, 100, 2048))
    if kind == "step":
        c.update(M=1, N=min(c["N"], 200000))
    if kind in ("load", "dual"):
        c.update(NL=1)
    if kind == "load":
        c.update(R=1, E=1, M=1)
    c["R"] = min(c["R"], c["L"] // 4)
    if kind in ("step", "grid", "dual", "noalloc"):
        most, field = MOST_TERMS[mode], 0
        # halve the sizes in turn until the case is no larger than the listed ones, its outputs included
        while _units(c) > most or c["M"] * c["E"] * c["K"] * c["R"] > 3.3e7:
            f = ("M", "R", "N", "K", "NL", "E")[field % 6]
            c[f] = max(1 if f != "N" else 300, c[f] // 2)
            field += 1
    if kind == "grid" and mode in ("fp32", "exact") and c["M"] * c["K"] * c["R"] * c["NL"] <= 4e6:
        c["S"] = rng.random() < 0.5
    return c


def _classes(case):
    """Sizes, supports and input lengths of the classes."""
    K, N, L = case["K"], case["N"], case["L"]
    k = np.arange(K)
    if not case["ragged"]:
        return np.full(K, N, np.int64), np.full(K, L, np.int32), np.zeros(K, np.int32)
    n = np.maximum(1, (N * 0.05 ** (k / max(1, K - 1))).astype(np.int64) + 3 * k)
    return n, (L - (k * 37) % (1 + L // 8)).astype(np.int32), ((k * 101) % (1 + L // 16)).astype(np.int32)


def _units(case):
    n, _, _ = _classes(case)
    cells = case["M"] * case["R"]
    if case["mode"] == "dual":
        return cells * case["E"] * case["K"]
    if case["mode"] == "envelope":
        return cells * case["NL"] * case["K"]
    return cells * case["NL"] * int(n.sum())


def _inputs(case, seed):
    """Samples on the GPU (lognormal output lengths, or 70 % lognormal and 30 % Pareto) and the grids."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, L, Lin = _classes(case)
    K = case["K"]
    med, sig = np.logspace(math.log10(0.00125 * case["L"]), math.log10(0.125 * case["L"]), K), np.linspace(0.6, 1.2, K)
    parts = []
    for k in range(K):
        z = torch.randn(int(n[k]), generator=g, device="cuda")
        if case["tail"]:
            body = torch.exp(math.log(200.0) + 0.7 * z)
            pareto = 500.0 * torch.rand(int(n[k]), generator=g, device="cuda").clamp_min(1e-7) ** (-1 / 1.3)
            x = torch.where(torch.rand(int(n[k]), generator=g, device="cuda") < 0.3, pareto, body)
        else:
            x = torch.exp(math.log(med[k]) + sig[k] * z)
        parts.append(x.clamp(1, float(L[k])).round().to(torch.int32))
    off = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    lo, hi = int(Lin.max()), int((Lin + L).min())
    every = case["R"] >= hi - lo + 1  # every integer reservation, or a grid up to the top of the domain
    r = np.arange(lo, lo + case["R"]) if every else lo + np.round((hi - lo) * np.arange(1, case["R"] + 1) / case["R"])
    rho = np.array([case["rho"]]) if case["M"] == 1 else np.logspace(0, math.log10(case["rho"]), case["M"])
    eps = np.concatenate([[0.0], np.logspace(0, 3, case["E"] - 1)]) if case["E"] > 1 else np.array([50.0])
    lam_hi = max(100.0, float(rho.max()))
    return {"K": K, "off": off, "x": torch.cat(parts), "L": L, "Lin": Lin, "r": r.astype(np.int32),
            "lam": np.logspace(-3, math.log10(lam_hi), case["NL"]), "eps": eps, "cp": rho, "cw": np.ones(case["M"]),
            "q": np.linspace(0.0, 1.0, case["F"]) if case["F"] > 1 else np.array([0.9])}


class _Context:
    """A context handle that is given back when the program drops it."""

    def __init__(self):
        self.h = kv.kvdro_create(torch.cuda.current_device())

    def __del__(self):
        kv.kvdro_destroy(self.h)


def prepare(case, seed):
    s = dict(_inputs(case, seed), case=case)
    K, M, E, R = case["K"], case["M"], case["E"], case["R"]
    f = torch.float32 if case["mode"] == "fp32" else torch.float64
    host = case["kind"] == "step"

    def out(shape, dtype):
        return torch.empty(shape, dtype=dtype, device="cpu" if host else "cuda")

    o = {}
    if case["kind"] in ("step", "load"):
        o["quant"] = out((K, case["F"]), torch.int32)
    if case["kind"] == "load":
        o["sorted"] = out((len(s["x"]),), torch.int32)
    else:
        o.update(r_idx=out((M, E, K), torch.int32), min_cost=out((M, E, K), f), fhat=out((M, E, K), torch.float64))
    if case["kind"] in ("grid", "noalloc"):
        o.update(cost=out((M, E, K, R), f), lam_idx=out((M, E, K, R), torch.int32))
    if case["kind"] == "dual":
        o.update(cost=out((M, E, K, R), f), gamma=out((M, E, K, R), f))
    if case["S"]:
        o["S"] = out((M, K, R, case["NL"]), f)
    s["out"] = o
    if case["kind"] != "noalloc":
        s["ctx"] = _Context()
    if case["kind"] in ("grid", "dual"):
        kv.kvdro_load_samples(s["ctx"].h, K, s["off"], s["x"], s["L"], s["Lin"], torch.cuda.current_stream())
    return s


def run(s):
    c, o, st = s["case"], s["out"], torch.cuda.current_stream()
    K, R, NL, E, M = c["K"], c["R"], c["NL"], c["E"], c["M"]
    if c["kind"] == "noalloc":
        kv.kvdro_eval_grid_noalloc(K, s["off"], s["x"], s["L"], s["Lin"], R, s["r"], NL, s["lam"], E, s["eps"], M,
                                   s["cp"], s["cw"], stream=st, **o)
        return o
    h = s["ctx"].h
    if c["kind"] in ("step", "load"):
        kv.kvdro_load_samples(h, K, s["off"], s["x"], s["L"], s["Lin"], st)
        kv.kvdro_quantiles(h, c["F"], s["q"], o["quant"], st)
    if c["kind"] == "load":
        kv.kvdro_sorted_samples(h, o["sorted"], st)
    elif c["kind"] == "dual":
        kv.kvdro_eval_dual(h, R, s["r"], E, s["eps"], M, s["cp"], s["cw"], stream=st, **o)
    else:
        kv.kvdro_eval_grid(h, MODES[c["mode"]], R, s["r"], NL, s["lam"], E, s["eps"], M, s["cp"], s["cw"], stream=st,
                           **{k: v for k, v in o.items() if k != "quant"})
    return o


def work(case):
    """Bytes: samples in, outputs out.  Flops: two per term in the per-term modes (a difference, a
    sum); ENVELOPE 10 per cell and 2 per cell and radius; the dual 2 per halving of the support and 10."""
    n, _, _ = _classes(case)
    total, rows = int(n.sum()), case["M"] * case["E"] * case["K"]
    es = 4 if case["mode"] == "fp32" else 8
    b = 4 * total
    if case["kind"] == "load":
        return {"bytes": 2 * b + 4 * case["K"] * case["F"], "flops": 2 * total}
    b += rows * (4 + es + 8)
    if case["kind"] in ("grid", "noalloc"):
        b += rows * case["R"] * (es + 4)
    if case["kind"] == "dual":
        b += rows * case["R"] * 16
    if case["S"]:
        b += case["M"] * case["K"] * case["R"] * case["NL"] * es
    units = _units(case)
    if case["mode"] == "dual":
        return {"bytes": b, "flops": units * (10 + 2 * math.ceil(math.log2(case["L"])))}
    if case["mode"] == "envelope":
        return {"bytes": b, "flops": units * (10 + 2 * case["E"])}
    return {"bytes": b, "flops": 2 * units}


def tolerance(case):
    if case["kind"] == "load":
        return "exact"
    # Four times the distances seen from exact() over the listed and some drawn cases: FP32 outputs,
    # rounded once, 6e-8; double sums 6e-14 at 5e5 samples, and they grow with the samples that a lane
    # adds in a row (twice that at 1e6); indices one in 1e5, on ties (more of a small array).
    if case["mode"] == "fp32":
        return {"rel": 2.4e-7, "max": 2.4e-7, "differ": 5e-4}
    return {"rel": 2.5e-13, "max": 5e-13, "differ": 5e-4}


# ---------------------------------------------------------------- the same results in 64 bits


def _key_argmin(cost, mode):
    """argmin over the last axis as documented: lowest index among equal FP32 costs, or among FP64
    costs equal in their upper 44 bits."""
    k = cost.float().view(torch.int32) if mode == "fp32" else cost.view(torch.int64) & ~0xFFFFF
    return (k == k.amin(-1, keepdim=True)).to(torch.int8).argmax(-1)


def _tails(x, L):
    """#{x < t} and sum of x < t for t in [0, L + 1]."""
    h = torch.bincount(x.long(), minlength=L + 1)[:L + 1]
    v = torch.arange(L + 1, device=x.device)
    zero = torch.zeros(1, dtype=torch.int64, device=x.device)
    return torch.cat([zero, h.cumsum(0)]), torch.cat([zero, (h * v).cumsum(0)])


def _sup_mean(cnt, sm, L, eta, lam, cp, cw):
    """Mean over the samples of the supremum, for broadcast eta and lam: phi = max(U, V) with
    V = c_w eta - min(lam, c_w) x below the point where they cross and U above it."""
    mu, nu = lam.clamp(max=cp), lam.clamp(max=cw)
    kap, d = mu + nu, cp * (L - eta) - mu * L - cw * eta
    t = torch.where(kap > 0, torch.floor(-d / kap.clamp_min(1e-300)) + 1, torch.where(d > 0, 0.0, L + 1.0))
    t = t.clamp(0, L + 1).long()
    below, s_below = cnt[t].double(), sm[t].double()
    n, above = cnt[-1].double(), (cnt[-1] - cnt[t]).double()
    dist = (L * (cnt[-1] - cnt[t]) - (sm[-1] - sm[t])).double()
    return (cw * eta * below - nu * s_below + cp * (L - eta) * above - mu * dist) / n, t


def exact(case, seed):
    s = _inputs(case, seed)
    K, M, E, R, NL = case["K"], case["M"], case["E"], case["R"], case["NL"]
    dev = s["x"].device  # (the largest dual cases take about 15 seconds)
    xs = [s["x"][int(s["off"][k]):int(s["off"][k + 1])] for k in range(K)]
    out = {}
    if case["kind"] in ("step", "load"):
        srt = [x.sort().values for x in xs]
        rank = [np.clip(np.ceil(s["q"] * len(x)), 1, len(x)).astype(np.int64) - 1 for x in xs]
        out["quant"] = torch.stack([v[torch.from_numpy(i).to(dev)] for v, i in zip(srt, rank)])
        if case["kind"] == "load":
            out["sorted"] = torch.cat(srt)
            return out
    lam, eps = torch.from_numpy(s["lam"]).to(dev), torch.from_numpy(s["eps"]).to(dev)
    cost = torch.empty((M, E, K, R), dtype=torch.float64, device=dev)
    lam_idx = torch.empty((M, E, K, R), dtype=torch.int32, device=dev)
    S_all = torch.empty((M, K, R, NL), dtype=torch.float64, device=dev) if case["S"] else None
    cdf = []
    for k in range(K):
        L = int(s["L"][k])
        cnt, sm = _tails(xs[k], L)
        eta = torch.from_numpy(s["r"]).to(dev).double() - float(s["Lin"][k])
        cdf.append(cnt[eta.long() + 1].double() / cnt[-1].double())
        for m in range(M):
            cp, cw = float(s["cp"][m]), float(s["cw"][m])
            if case["kind"] == "dual":
                cost[m, :, k] = _dual(cnt, sm, L, eta, eps, cp, cw)
                continue
            S, _ = _sup_mean(cnt, sm, L, eta[:, None], lam[None, :], cp, cw)
            if S_all is not None:
                S_all[m, k] = S
            for e in range(E):
                v = lam * eps[e] + S
                cost[m, e, k] = v.amin(-1)
                lam_idx[m, e, k] = (v == v.amin(-1, keepdim=True)).to(torch.int8).argmax(-1).int()
    r_idx = _key_argmin(cost, case["mode"])
    out["r_idx"] = r_idx.int()
    out["min_cost"] = cost.gather(-1, r_idx[..., None])[..., 0]
    out["fhat"] = torch.stack(cdf)[torch.arange(K, device=dev), r_idx]
    if case["kind"] in ("grid", "noalloc"):
        out.update(cost=cost, lam_idx=lam_idx)
    if case["kind"] == "dual":
        out.update(cost=cost, gamma=None)  # any gamma between two equal kinks is a minimiser
    if S_all is not None:
        out["S"] = S_all
    return out


def _dual(cnt, sm, L, eta, eps, cp, cw):
    """min over gamma >= 0 of gamma eps + S(eta, gamma), a convex function: bisection on the sign of
    its right derivative over the ordered bit patterns of the doubles in [0, max(c_p, c_w)]."""
    e, eps = eta[None, :], eps[:, None]
    n = cnt[-1].double()
    shape = torch.broadcast_shapes(e.shape, eps.shape)
    lo = torch.zeros(shape, dtype=torch.int64, device=eta.device)
    hi = torch.full(shape, max(cp, cw), dtype=torch.float64, device=eta.device).view(torch.int64)

    def rising(g):
        _, t = _sup_mean(cnt, sm, L, e, g, cp, cw)
        drop = (g < cw) * sm[t] + (g < cp) * (L * (cnt[-1] - cnt[t]) - (sm[-1] - sm[t]))
        return eps * n >= drop.double()

    at0 = rising(lo.view(torch.float64))
    hi = torch.where(at0, lo, hi)
    for _ in range(63):
        mid = lo + torch.div(hi - lo, 2, rounding_mode="floor")
        up = rising(mid.view(torch.float64))
        lo, hi = torch.where(up, lo, mid), torch.where(up, mid, hi)
    best = torch.minimum(*(g * eps + _sup_mean(cnt, sm, L, e, g, cp, cw)[0]
                           for g in (lo.view(torch.float64), hi.view(torch.float64))))
    i = eta.long()  # the empirical cost, the value at radius 0, bounds it from below
    up_n, up_s = (cnt[-1] - cnt[i + 1]).double(), (sm[-1] - sm[i + 1]).double()
    emp = (cw * (eta * cnt[i + 1].double() - sm[i + 1].double()) + cp * (up_s - eta * up_n)) / n
    return torch.maximum(best, emp[None, :])
