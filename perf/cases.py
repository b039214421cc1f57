"""Workloads that time this library through its public entry points.

Each case is one thing a program that factors sparse count tensors asks of the
library: Phi^(n) or MTTKRP of a resident tensor, a solve of some outer
iterations of CP-APR MU from a given start, a batched solve of many small
tensors, or bringing a new tensor in from host memory.  Tensors are drawn on
the GPU with the statistics of `paper_2307_03276_gb300/synth.py` (Zipf or
uniform modes with scattered heavy rows, distinct coordinates in random order,
Poisson or geometric counts; U(0,1) factors) at the sizes of its specs.

A case is a dict of plain values:
  kind    phi | mttkrp | solve | batch | load
  dims    "I1xI2x..", modes "z1.2,u,.." (Zipf exponent or uniform, per mode)
  values  "poisson1.0" (Poisson + 1) or "geometric0.5" (1, 2, ..)
  nnz, rank, precision ("f64" or "f32"), outer (outer iterations of a solve)
  mode    the one mode of a phi case, -1 for every mode in turn
  pi      "auto" (the library's choice) or "fused" (a caller short of memory)
  count, spec_seed   a batch's number of tensors and the seed of its shapes
The FP32 form computes in single precision; its results are returned as
float32 (a Phi entry is a float32 value widened by the interface).
"""
import ctypes
import math
import random

import torch

from paper_2307_03276_gb300 import cpapr

TOL = 1e-4       # KKT tolerance of the solves
MAX_INNER = 10   # inner iterations per mode and outer iteration
KAPPA, KAPPA_TOL, EPS = 0.01, 1e-10, 1e-10  # the library's documented defaults


# ---- cases -----------------------------------------------------------------

def _case(name, kind, dims, modes, values, nnz, rank, precision, **more):
    c = {"name": name, "kind": kind, "dims": "x".join(str(d) for d in dims), "modes": modes, "values": values,
         "nnz": nnz, "rank": rank, "precision": precision}
    c.update(more)
    return c


def listed():
    small = ((100, 80, 60), "u,u,u", "poisson1.0", 10_000, 10)
    way3 = ((100_000, 100_000, 1_000), "z1.2,z1.2,z1.2", "poisson2.0", 10_000_000, 32)
    way4 = ((200_000, 200_000, 10_000, 365), "z1.1,z1.1,u,u", "geometric0.5", 50_000_000, 16)
    way5 = ((50_000, 49_999, 5_001, 1_000, 24), "z1.3,z1.3,z1.3,z1.3,z1.3", "poisson1.0", 3_000_017, 33)
    batch = {"dims": "", "modes": "z1.2,z1.2,z1.2", "values": "poisson1.0", "nnz": 0, "rank": 0, "count": 64,
             "spec_seed": 1004, "outer": 2}
    return [
        # one Phi of a small tensor: the latency of a call
        _case("phi_small_f64", "phi", *small, "f64", mode=0),
        # a short solve of the same tensor: hundreds of tiny dependent launches
        _case("solve_small_f64", "solve", *small, "f64", outer=10, pi="auto"),
        # Phi of every mode of a mid-size 5-way tensor, odd sizes, a rank that is padded
        _case("phi_5way_odd_f64", "phi", *way5, "f64", mode=-1),
        # MTTKRP of every mode (the first step of an ALS or gradient code on the same tensor)
        _case("mttkrp_4way_f64", "mttkrp", *way4, "f64"),
        _case("mttkrp_3way_f32", "mttkrp", *way3, "f32"),
        # an outer iteration of the large single tensors, in both precisions
        _case("solve_3way_f64", "solve", *way3, "f64", outer=1, pi="auto"),
        _case("solve_3way_f32", "solve", *way3, "f32", outer=1, pi="auto"),
        _case("solve_4way_f64", "solve", *way4, "f64", outer=1, pi="auto"),
        _case("solve_4way_f32", "solve", *way4, "f32", outer=1, pi="auto"),
        # many small uneven tensors together (one per user, site or day)
        dict(batch, name="batch64_f64", kind="batch", precision="f64"),
        dict(batch, name="batch64_f32", kind="batch", precision="f32"),
        # a new tensor arrives in pinned host memory: index it, set a model, take its first Phi
        _case("load_3way_f64", "load", *way3, "f64", mode=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["phi", "phi", "mttkrp", "solve", "solve", "solve", "batch", "load"])
    precision = rng.choice(["f64", "f32"])
    if kind == "batch":
        return {"kind": "batch", "dims": "", "modes": "z1.2,z1.2,z1.2", "values": "poisson1.0", "nnz": 0, "rank": 0,
                "count": _log_int(rng, 4, 64), "spec_seed": rng.randrange(1 << 20), "outer": rng.randint(1, 2),
                "precision": precision}
    n = rng.choice([2, 3, 3, 4, 4, 5, 6])
    rank = rng.choice([rng.randint(1, 64), 8, 16, 32, 64])
    nnz = min(_log_int(rng, 1e3, 2e7), 320_000_000 // rank)
    dims, modes = [], []
    for m in range(n):
        dims.append(_log_int(rng, 20, 200_000) if m else _log_int(rng, 200, 200_000))
        modes.append(rng.choice(["u", "z1.1", "z1.2", "z1.3"]))
    # distinct Zipf coordinates fill a small part of a space: keep at most 2% of its cells
    while math.prod(dims) < 50 * nnz:
        m = min(range(n), key=lambda k: dims[k])
        dims[m] = dims[m] * 3 + rng.randint(0, 2)
    while math.prod(dims) >= 1 << 61:  # a cell's number is an int64
        m = max(range(n), key=lambda k: dims[k])
        dims[m] //= 2
    c = {"kind": kind, "dims": "x".join(map(str, dims)), "modes": ",".join(modes),
         "values": rng.choice(["poisson1.0", "poisson2.0", "geometric0.5"]), "nnz": nnz, "rank": rank,
         "precision": precision}
    if kind == "phi":
        c["mode"] = rng.choice([-1, rng.randrange(n)])
    if kind == "load":
        c["mode"] = rng.randrange(n)
    if kind == "solve":
        c["outer"] = _log_int(rng, 1, 10) if nnz < 200_000 else rng.randint(1, 2) if nnz < 5_000_000 else 1
        c["pi"] = rng.choice(["auto", "auto", "auto", "fused"])
    return c


def _batch_shapes(case):
    """(dims, nnz, rank) of a batch's tensors: log-uniform sizes, a tenth of the cells at most."""
    rng = random.Random(int(case["spec_seed"]))
    shapes = []
    for _ in range(case["count"]):
        dims = (_log_int(rng, 50, 20_000), _log_int(rng, 50, 20_000), _log_int(rng, 50, 500))
        nnz = min(_log_int(rng, 1e3, 1e6), math.prod(dims) // 10)
        shapes.append((dims, nnz, rng.choice([8, 16, 32])))
    return shapes


# ---- inputs ----------------------------------------------------------------

def _coordinates(dims, modes, nnz, gen, dev):
    """[N, nnz] distinct int64 coordinates in random order."""
    tables = []
    for d, kind in zip(dims, modes.split(",")):
        if kind == "u":
            tables.append(None)
            continue
        w = torch.arange(1, d + 1, dtype=torch.float64, device=dev) ** (-float(kind[1:]))
        cdf = torch.cumsum(w, 0)
        # heavy rows are scattered over the mode
        tables.append((cdf / cdf[-1], torch.randperm(d, generator=gen, device=dev)))
    keys = torch.empty(0, dtype=torch.int64, device=dev)
    want = int(nnz * 1.15) + 64
    for _ in range(200):
        lin = torch.zeros(want, dtype=torch.int64, device=dev)
        for d, t in zip(dims, tables):
            u = torch.rand(want, generator=gen, device=dev, dtype=torch.float64)
            k = (u * d).long() if t is None else torch.searchsorted(t[0], u, right=True)
            k.clamp_(max=d - 1)
            lin.mul_(d).add_(k if t is None else t[1][k])
        keys = torch.unique(torch.cat([keys, lin]))
        if keys.numel() >= nnz:
            break
        want = 3 * (nnz - keys.numel()) + 1024
    else:
        raise RuntimeError("could not draw enough distinct coordinates")
    keys = keys[torch.randperm(keys.numel(), generator=gen, device=dev)[:nnz]]
    idx = torch.empty((len(dims), nnz), dtype=torch.int64, device=dev)
    for m in range(len(dims) - 1, -1, -1):
        idx[m] = keys % dims[m]
        keys = keys // dims[m]
    return idx


def _counts(values, nnz, gen, dev):
    if values.startswith("poisson"):
        rate = torch.full((nnz,), float(values[7:]), dtype=torch.float64, device=dev)
        return torch.poisson(rate, generator=gen) + 1.0
    u = torch.rand(nnz, generator=gen, device=dev, dtype=torch.float64)
    return torch.clamp(torch.floor(torch.log1p(-u) / math.log1p(-float(values[9:]))), max=63.0) + 1.0


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _tensor(dims, modes, values, nnz, rank, gen, dev):
    idx = _coordinates(dims, modes, nnz, gen, dev)
    vals = _counts(values, nnz, gen, dev)
    factors = [torch.rand((d, rank), generator=gen, device=dev, dtype=torch.float64) for d in dims]
    lam = 0.5 + torch.rand(rank, generator=gen, device=dev, dtype=torch.float64)
    return {"dims": dims, "rank": rank, "idx": idx, "vals": vals, "lam": lam, "factors": factors}


def _inputs(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 17)
    if case["kind"] == "batch":
        return [_tensor(d, case["modes"], case["values"], z, r, gen, dev) for d, z, r in _batch_shapes(case)]
    return _tensor(_dims(case), case["modes"], case["values"], case["nnz"], case["rank"], gen, dev)


def _options(case):
    o = {"precision": cpapr.CPAPR_FP32 if case["precision"] == "f32" else cpapr.CPAPR_FP64}
    if case.get("pi", "auto") == "fused":
        o["pi_mode"] = cpapr.CPAPR_PI_FUSED
    return o


def _context(case, x):
    return cpapr.Tensor(x["dims"], [x["idx"][m] for m in range(len(x["dims"]))], x["vals"], x["rank"], **_options(case))


def _model_buffers(tensors):
    """One flat device buffer for the models of these tensors, and each one's
    addresses in it (lambda, then the factors)."""
    sizes = [n for x in tensors for n in [x["rank"]] + [d * x["rank"] for d in x["dims"]]]
    flat = torch.zeros(sum(sizes), dtype=torch.float64, device="cuda")
    parts = iter(torch.split(flat, sizes))
    where = []
    for x in tensors:
        lam = next(parts).data_ptr()
        where.append((lam, (ctypes.c_void_p * len(x["dims"]))(*[next(parts).data_ptr() for _ in x["dims"]])))
    return flat, where


def prepare(case, seed):
    x = _inputs(case, seed)
    torch.cuda.synchronize()
    kind = case["kind"]
    if kind == "batch":
        ctxs = [_context(case, t) for t in x]
        models = [(t["lam"], t["factors"]) for t in x]
        flat, where = _model_buffers(x)
        return {"case": case, "tensors": ctxs, "models": models, "out": flat, "where": where}
    if kind == "load":
        host_idx = [x["idx"][m].cpu().pin_memory() for m in range(len(x["dims"]))]
        host_vals = x["vals"].cpu().pin_memory()
        out = torch.zeros((x["dims"][case["mode"]], x["rank"]), dtype=torch.float64, device="cuda")
        return {"case": case, "dims": x["dims"], "rank": x["rank"], "idx": host_idx, "vals": host_vals,
                "model": (x["lam"], x["factors"]), "out": out}
    t = _context(case, x)
    state = {"case": case, "tensor": t, "model": (x["lam"], x["factors"])}
    if kind == "solve":
        state["out"], state["where"] = _model_buffers([x])
    else:
        t.set_model(x["lam"], x["factors"])
        modes = range(len(x["dims"])) if case.get("mode", -1) < 0 else [case["mode"]]
        state["out"] = {m: torch.zeros((x["dims"][m], x["rank"]), dtype=torch.float64, device="cuda") for m in modes}
    torch.cuda.synchronize()
    return state


# ---- one pass --------------------------------------------------------------

def _typed(case, t):
    return t.float() if case["precision"] == "f32" else t


def _fetch(tensor, where):
    """The model into device buffers, through the C interface (it takes device pointers)."""
    st = cpapr.load().cpapr_get_model(tensor.ctx, *where)
    if st != 0:
        raise cpapr.CpaprError(st, cpapr.cpapr_last_error(tensor.ctx))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "phi":
        return [_typed(case, state["tensor"].phi(m, out=o)) for m, o in state["out"].items()]
    if kind == "mttkrp":
        return [_typed(case, state["tensor"].mttkrp(m, out=o)) for m, o in state["out"].items()]
    if kind == "load":
        with cpapr.Tensor(state["dims"], state["idx"], state["vals"], state["rank"], **_options(case)) as t:
            t.set_model(*state["model"])
            return _typed(case, t.phi(case["mode"], out=state["out"]))
    if kind == "solve":
        t = state["tensor"]
        t.set_model(*state["model"])
        res = t.mu_solve(tol=TOL, max_outer=case["outer"], max_inner=MAX_INNER)
        _fetch(t, state["where"][0])
        return {"model": _typed(case, state["out"]), "loglik": res["loglik"], "kkt": res["kkt_viol"],
                "inner": res["total_inner"]}
    for t, m in zip(state["tensors"], state["models"]):
        t.set_model(*m)
    res = cpapr.cpapr_batch_mu_solve([t.ctx for t in state["tensors"]], tol=TOL, max_outer=case["outer"],
                                     max_inner=MAX_INNER)
    for t, w in zip(state["tensors"], state["where"]):
        _fetch(t, w)
    return {"models": _typed(case, state["out"]),
            "loglik": torch.tensor([r["loglik"] for r in res]),
            "inner": torch.tensor([r["total_inner"] for r in res])}


# ---- what a pass cannot do without -----------------------------------------

def _phi_work(dims, nnz, rank, b, modes):
    """Coordinates, counts, factors and B read once and Phi written once per
    evaluation; per nonzero a Khatri-Rao row, a dot product, a division and a
    scaled addition."""
    n = len(dims)
    by = fl = 0
    for m in modes:
        by += nnz * (4 * (n - 1) + b) + 4 * dims[m] + b * rank * (sum(dims) + dims[m])
        fl += nnz * ((n + 2) * rank + 2)
    return by, fl


def _solve_work(dims, nnz, rank, b, outer):
    n = len(dims)
    by, fl = _phi_work(dims, nnz, rank, b, range(n))
    evals = outer * MAX_INNER
    # B <- B * Phi after each evaluation; the start and the result, FP64
    return (by + 3 * b * rank * sum(dims)) * evals + 16 * rank * (sum(dims) + 1), (fl + rank * sum(dims)) * evals


def work(case):
    b = 4 if case["precision"] == "f32" else 8
    kind = case["kind"]
    if kind == "batch":
        parts = [_solve_work(d, z, r, b, case["outer"]) for d, z, r in _batch_shapes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    dims, nnz, rank = _dims(case), case["nnz"], case["rank"]
    n = len(dims)
    if kind == "solve":
        by, fl = _solve_work(dims, nnz, rank, b, case["outer"])
    elif kind == "phi":
        by, fl = _phi_work(dims, nnz, rank, b, range(n) if case["mode"] < 0 else [case["mode"]])
    elif kind == "mttkrp":
        by, fl = _phi_work(dims, nnz, rank, b, range(n))
        by, fl = by - b * rank * sum(dims), n * nnz * n * rank
    else:
        by, fl = _phi_work(dims, nnz, rank, b, [case["mode"]])
        by += nnz * (8 * n + 8) + n * nnz * (4 * (n - 1) + b) + 8 * rank * sum(dims)  # the COO in, a layout per mode out
    return {"bytes": by, "flops": fl}


# ---- the same in 64 bits, with plain torch ---------------------------------

def _exact_phi(x, factors, n, B):
    """Phi^(n) (B given) or the MTTKRP (B None), nonzeros in chunks."""
    nnz, rank = x["vals"].numel(), x["rank"]
    out = torch.zeros((x["dims"][n], rank), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 28) // rank)
    for lo in range(0, nnz, step):
        hi = min(nnz, lo + step)
        pi = None
        for m, A in enumerate(factors):
            if m != n:
                row = A[x["idx"][m, lo:hi]]
                pi = row if pi is None else pi.mul_(row)
        v = x["vals"][lo:hi]
        if B is not None:
            s = (B[x["idx"][n, lo:hi]] * pi).sum(1)
            v = v / torch.clamp(s, min=EPS)
        out.index_add_(0, x["idx"][n, lo:hi], pi.mul_(v[:, None]))
    return out


def _exact_solve(x, outer):
    n = len(x["dims"])
    factors = [A.clone() for A in x["factors"]]
    lam = x["lam"].clone()
    prev = [torch.zeros_like(A) for A in factors]
    total, kkt = 0, 0.0
    for k in range(outer):
        first, kkt = True, 0.0
        for m in range(n):
            shift = torch.where((factors[m] < KAPPA_TOL) & (prev[m] > 1.0), KAPPA, 0.0) if k else 0.0
            B = (factors[m] + shift) * lam
            for l in range(MAX_INNER):
                phi = _exact_phi(x, factors, m, B)
                total += 1
                viol = float(torch.minimum(B, 1.0 - phi).abs().max())
                if viol < TOL:
                    break
                B = B * phi
                first = False
            prev[m] = phi
            kkt = max(kkt, viol)
            lam = B.sum(0)
            factors[m] = torch.where(lam > 0, B / lam, factors[m])
        if first:
            break
    ll, nnz = 0.0, x["vals"].numel()
    step = max(1, (1 << 28) // x["rank"])
    for lo in range(0, nnz, step):
        hi = min(nnz, lo + step)
        p = lam.expand(hi - lo, -1).clone()
        for m, A in enumerate(factors):
            p.mul_(A[x["idx"][m, lo:hi]])
        ll += float((x["vals"][lo:hi] * torch.log(p.sum(1))).sum())
    mass = lam.clone()
    for A in factors:
        mass = mass * A.sum(0)
    return torch.cat([lam] + [A.reshape(-1) for A in factors]), ll - float(mass.sum()), kkt, total


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        got = [_exact_solve(t, case["outer"]) for t in x]
        return {"models": torch.cat([g[0] for g in got]), "loglik": torch.tensor([g[1] for g in got]), "inner": None}
    if kind == "solve":
        model, ll, kkt, _ = _exact_solve(x, case["outer"])
        return {"model": model, "loglik": ll, "kkt": kkt, "inner": None}
    if kind == "load":
        m = case["mode"]
        return _exact_phi(x, x["factors"], m, x["factors"][m] * x["lam"])
    modes = range(len(x["dims"])) if case.get("mode", -1) < 0 else [case["mode"]]
    return [_exact_phi(x, x["factors"], m, x["factors"][m] * x["lam"] if kind == "phi" else None) for m in modes]
