"""Timed cases of the Digital Annealer library: whole calls of its public entry points over the
range of sizes, coupling types and options that its users run.

Every case is one call (or the few calls of one task) as a program makes it:

- "anneal":  da_anneal on a context kept by the program, host schedule in, host results out;
- "device":  da_anneal_async on the program's stream, schedule and results in device memory;
- "static":  da_anneal_static, the allocation-free int8 anneal on device arrays;
- "oneshot": a new QUBO from host memory: da_create, da_anneal, da_destroy;
- "ptda":    da_pt, parallel tempering with the exchange after every sweep;
- "batch":   da_batch_anneal, many instances of mixed sizes and coupling types in one call;
- "serve":   the request loop: a burst of da_submit, then da_poll for every result;
- "fields":  da_field_recompute and da_energy of many host states.

Coupling types: "int8" (bimodal couplings), "fp32" (Gaussian), "int16" (Gaussian scaled to the
16-bit fixed-point precision with da_quantize).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_08815_gb300 import binding as da
from paper_1806_08815_gb300 import instances


def listed():
    return [
        # a first look at a tiny problem: what one call costs before any annealing matters
        dict(name="call_33_int8", kind="anneal", dtype="int8", N=33, R=4, T=200, inc=1.0),
        # the small complete-graph benchmark workload
        dict(name="sk_64_int8", kind="anneal", dtype="int8", N=64, R=64, T=10_000, inc=1.0),
        # the 2D spin glass on a 32 x 32 torus, held dense: few replicas, a long geometric schedule
        dict(name="torus_1024_fp32", kind="anneal", dtype="fp32", N=1024, R=128, T=100_000, inc=0.5, torus=True),
        # the headline anneal: one large instance, replicas enough to fill the GPU
        dict(name="sk_1024_fp32", kind="anneal", dtype="fp32", N=1024, R=1024, T=200_000, inc=0.0),
        # the 16-bit fixed-point precision of the annealing hardware, ragged size, results kept on the device
        dict(name="fixed_1000_int16", kind="device", dtype="int16", N=1000, R=500, T=20_000, inc=0.0),
        # the allocation-free form in a program that owns the memory, ragged size
        dict(name="static_200_int8", kind="static", dtype="int8", N=200, R=512, T=10_000, inc=1.0),
        # a new middle-sized QUBO solved once: upload, build, anneal, results
        dict(name="oneshot_3000_int8", kind="oneshot", dtype="int8", N=3000, R=32, T=20_000, inc=1.0),
        # the largest instance with the replicas of a served request, results kept on the device
        dict(name="sk_8192_fp32", kind="device", dtype="fp32", N=8192, R=32, T=8192, inc=0.0),
        # parallel tempering: 32 ladders of 32 temperatures
        dict(name="ptda_512_int8", kind="ptda", dtype="int8", N=512, K=32, L=32, sweeps=50, adapt=0),
        # an instance set solved together, sizes and coupling types mixed, ragged ones among them
        dict(name="batch_64_mixed", kind="batch", sizes="64,128,250,256,500,512,1000,1024", n=64, R=64, T=5_000),
        # a burst at the request loop, sizes log-uniform, both coupling types
        dict(name="serve_8_mixed", kind="serve", lo=256, hi=4096, n=8, R=32, T=10_000),
        # fields and energies of many states (temperature grids, checks of stored solutions)
        dict(name="fields_2048_fp32", kind="fields", dtype="fp32", N=2048, R=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _anneal_size(rng, n_lo, n_hi, r_hi):
    """N and R log-uniform, and a step count whose trials stay far below the largest listed case."""
    N = _log_int(rng, n_lo, n_hi)
    if rng.random() < 0.25:                       # powers of two are common in use too
        N = 1 << round(math.log2(N))
        N = max(n_lo, min(n_hi, N))
    R = _log_int(rng, 1, min(r_hi, max(8, (1 << 20) // N)))
    # bounded by the trials (throughput) and by the step count (latency of few replicas)
    T = _log_int(rng, 200, 20_000)
    return N, R, max(200, min(T, int(3e10 / (N * max(R, 64)))))


def draw(rng):
    kind = rng.choice(["anneal", "anneal", "device", "static", "oneshot", "ptda", "batch", "serve", "fields"])
    if kind in ("anneal", "device"):
        N, R, T = _anneal_size(rng, 33, 8192, 2048)
        dtype = rng.choice(["int8", "fp32", "fp32", "int16"])
        c = dict(kind=kind, dtype=dtype, N=N, R=R, T=T, inc=rng.choice([0.0, 0.5, 1.0]))
        if dtype == "fp32" and N <= 1024 and rng.random() < 0.3:
            L = max(6, int(math.sqrt(N)))
            c.update(N=L * L, torus=True)
        return c
    if kind == "static":
        N, R, T = _anneal_size(rng, 33, 1024, 1024)
        return dict(kind=kind, dtype="int8", N=N, R=R, T=T, inc=rng.choice([0.0, 1.0]))
    if kind == "oneshot":
        N, R, T = _anneal_size(rng, 128, 6000, 128)
        return dict(kind=kind, dtype=rng.choice(["int8", "fp32"]), N=N, R=R, T=T, inc=rng.choice([0.0, 1.0]))
    if kind == "ptda":
        N = _log_int(rng, 48, 1500)
        return dict(kind=kind, dtype=rng.choice(["int8", "fp32", "int16"]), N=N, K=rng.randint(2, 40),
                    L=rng.randint(1, 32), sweeps=rng.randint(3, max(4, min(60, 20_000 // N))),
                    adapt=rng.choice([0, 0, 5]))
    if kind == "batch":
        sizes = sorted(_log_int(rng, 40, 1024) for _ in range(rng.randint(2, 8)))
        return dict(kind=kind, sizes=",".join(map(str, sizes)), n=rng.randint(4, 64), R=_log_int(rng, 8, 100),
                    T=_log_int(rng, 500, 5_000))
    if kind == "serve":
        return dict(kind=kind, lo=rng.randint(64, 512), hi=rng.randint(1024, 4096), n=rng.randint(1, 8),
                    R=_log_int(rng, 4, 64), T=_log_int(rng, 500, 10_000))
    return dict(kind="fields", dtype=rng.choice(["int8", "fp32", "fp32", "int16"]), N=_log_int(rng, 64, 6000),
                R=_log_int(rng, 1, 2048))


# ---- inputs -----------------------------------------------------------------------------------

_DT = {"int8": da.DA_INT8, "fp32": da.DA_FP32, "int16": da.DA_INT16}


def _couplings(dtype, N, seed, torus=False):
    """Ising couplings J (N x N, upper triangle, fp64 on the GPU): bimodal or N(0, 1)/sqrt(N) on the
    complete graph, N(0, 1) on the edges of a torus."""
    g = torch.Generator("cuda").manual_seed(seed)
    if torus:
        L = math.isqrt(N)
        i = torch.arange(N, device="cuda").view(L, L)
        a = i.flatten().repeat(2)
        b = torch.cat([i.roll(-1, 1).flatten(), i.roll(-1, 0).flatten()])
        J = torch.zeros(N, N, dtype=torch.float64, device="cuda")
        w = torch.randn(2 * N, generator=g, device="cuda").double()
        J[torch.minimum(a, b), torch.maximum(a, b)] = w
        return J
    if dtype == "int8":
        J = torch.randint(0, 2, (N, N), generator=g, device="cuda").mul_(2).sub_(1).double()
    else:
        J = torch.randn(N, N, generator=g, device="cuda").div_(math.sqrt(N)).double()
    return J.triu_(1)


def _qubo(dtype, N, seed, torus=False):
    """Host QUBO of the couplings with s = 2x - 1 (int32 for "int8", else fp32), row-major, upper triangle."""
    J = _couplings(dtype, N, seed, torus)
    row = J.sum(0) + J.sum(1)
    Q = -4.0 * J
    Q.diagonal().copy_(2.0 * row)
    return Q.to(torch.int32 if dtype == "int8" else torch.float32).cpu().numpy()


def _schedule(dtype, T, torus=False):
    if torus:
        return instances.beta_geometric(0.1, 5.0, T)
    return instances.beta_linear(0.05, 3.0, T) if dtype == "int8" else instances.beta_linear(0.1, 10.0, T)


def _problem(dtype, N, seed, torus=False):
    """(host QUBO in the library's input form, da dtype, factor on the energies)."""
    Q = _qubo(dtype, N, seed, torus)
    if dtype != "int16":
        return Q, _DT[dtype], 1.0
    Qi, scale = da.da_quantize(Q)
    return Qi, da.DA_INT16, scale


def _recompute(dtype):
    return 1024 if dtype == "fp32" else 0     # the period used throughout for real couplings


def _device_outputs(N, R):
    f = lambda: torch.zeros(R, dtype=torch.float64, device="cuda")
    x = lambda: torch.zeros((R, da.da_words(N)), dtype=torch.int32, device="cuda")
    return dict(final_E=f(), best_E=f(), final_x=x(), best_x=x(), max_drift=f(),
                flips=torch.zeros(R, dtype=torch.int64, device="cuda"))


def _mixed(case):
    """(dtype, N) of the items of a mixed set: sizes in turn or log-uniform, coupling types alternating."""
    if case["kind"] == "batch":
        sizes = [int(s) for s in case["sizes"].split(",")]
        ns = [sizes[(i // 2) % len(sizes)] for i in range(case["n"])]
    else:
        # log-uniform: the midpoints of n equal intervals, arriving in a fixed shuffled order
        n, span = case["n"], math.log(case["hi"] / case["lo"])
        ns = [int(round(case["lo"] * math.exp(span * (i + 0.5) / n))) for i in range(n)]
        ns = [ns[k] for k in np.random.default_rng(n).permutation(n)]
    return [("int8" if i % 2 == 0 else "fp32", N) for i, N in enumerate(ns)]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind in ("batch", "serve"):
        items = []
        for i, (dtype, N) in enumerate(_mixed(case)):
            Q = _qubo(dtype, N, seed * 1009 + i)
            items.append(dict(beta=_schedule(dtype, case["T"]), offset_inc=1.0 if dtype == "int8" else 0.0,
                              replicas=case["R"], seed=seed + i, recompute_every=_recompute(dtype)))
            items[-1].update({"ctx": da.da_create(Q)} if kind == "batch" else {"Q": Q})
        st["items"] = items
        if kind == "serve":
            st["server"] = da.Server(120 << 30, 1024)
        return st
    dtype, N = case["dtype"], case["N"]
    Q, dt, scale = _problem(dtype, N, seed, case.get("torus", False))
    if kind == "oneshot":
        st.update(Q=Q, dt=dt)
    elif kind == "static":
        ldw = da.da_static_pitch(N)
        W = np.zeros((N, ldw), np.int8)
        U = np.triu(Q, 1)
        W[:, :N] = U + U.T
        st.update(W=torch.from_numpy(W).cuda(), diag=torch.from_numpy(np.diag(Q).copy()).cuda(), ldw=ldw)
    else:
        st["ctx"] = da.da_create(Q, dt)
    if kind == "ptda":
        st["betas"] = (instances.beta_geometric(0.2, 5.0, case["K"]) / scale).astype(np.float32)
        return st
    if kind == "fields":
        x = np.random.default_rng(seed).integers(0, 2, (case["R"], da.da_words(N) * 32), dtype=np.uint8)
        x[:, N:] = 0
        st["x"] = np.packbits(x, axis=1, bitorder="little").view(np.uint32)
        return st
    st["beta"] = (_schedule(dtype, case["T"], case.get("torus", False)) / scale).astype(np.float32)
    if kind in ("device", "static"):
        st.update(beta=torch.from_numpy(st["beta"]).cuda(), out=_device_outputs(N, case["R"]))
    return st


# ---- one pass ---------------------------------------------------------------------------------

_TIMES = ("elapsed_s", "latency_s")


def _results(out):
    return {k: v for k, v in out.items() if k not in _TIMES}


def _joined(outs):
    """The results of several instances, each kind of result as one array."""
    return {k: np.concatenate([o[k].ravel() for o in outs]) for k in _results(outs[0])}


def run(st):
    c, seed = st["case"], st["seed"]
    kind = c["kind"]
    if kind == "anneal":
        return _results(da.da_anneal(st["ctx"], st["beta"], c["inc"], c["R"], seed, _recompute(c["dtype"])))
    if kind == "device":
        da.da_anneal_async(st["ctx"], st["beta"], c["T"], c["inc"], c["R"], seed, _recompute(c["dtype"]), st["out"],
                           torch.cuda.current_stream())
        return st["out"]
    if kind == "static":
        da.da_anneal_static(st["W"], st["diag"], c["N"], st["ldw"], st["beta"], c["T"], c["inc"], c["R"], seed,
                            st["out"], torch.cuda.current_stream())
        return st["out"]
    if kind == "oneshot":
        ctx = da.da_create(st["Q"], st["dt"])
        out = da.da_anneal(ctx, st["beta"], c["inc"], c["R"], seed, _recompute(c["dtype"]))
        da.da_destroy(ctx)
        return _results(out)
    if kind == "ptda":
        return _results(da.da_pt(st["ctx"], st["betas"], c["sweeps"], c["L"], seed, adapt_every=c["adapt"],
                                 adapt_sweeps=c["sweeps"] // 2))
    if kind == "batch":
        outs, _ = da.da_batch_anneal(st["items"])
        return _joined(outs)
    if kind == "serve":
        reqs = [da.da_submit(st["server"], **it) for it in st["items"]]
        return _joined([da.da_poll(r, 600_000_000) for r in reqs])
    return dict(fields=da.da_field_recompute(st["ctx"], st["x"]), energy=da.da_energy(st["ctx"], st["x"]))


# ---- what a pass cannot do without ------------------------------------------------------------

def _anneal_work(N, R, T):
    words = (N + 31) // 32
    # in: the couplings and linear terms once, the schedule; out: two states, four 8-byte results per replica
    data = 4 * N * (N + 1) // 2 + 4 * T + R * (8 * words + 32)
    # per trial: Delta E, its product with beta, the comparison, and the field's fused update
    return dict(bytes=data, flops=5 * R * T * N)


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        parts = [_anneal_work(N, case["R"], case["T"]) for _, N in _mixed(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N = case["N"]
    if kind == "ptda":
        return _anneal_work(N, case["K"] * case["L"], case["sweeps"] * N)
    if kind == "fields":
        R = case["R"]
        return dict(bytes=4 * N * (N + 1) // 2 + R * (4 * ((N + 31) // 32) + 4 * N + 8), flops=2 * N * N * R + 3 * N * R)
    return _anneal_work(N, case["R"], case["T"])


# ---- reference in 64 bits ---------------------------------------------------------------------

def exact(case, seed):
    """Fields and energies are functions of the inputs alone; an anneal's results are those of its
    own trajectory of decisions, which has no value apart from the arithmetic that defines it."""
    if case["kind"] != "fields":
        return None
    N = case["N"]
    # the QUBO the library was given (for "int16" its quantized integers), in 64 bits
    Q = torch.from_numpy(_problem(case["dtype"], N, seed)[0]).cuda().double().triu()
    x = np.random.default_rng(seed).integers(0, 2, (case["R"], (N + 31) // 32 * 32), dtype=np.uint8)[:, :N]
    X = torch.from_numpy(x).cuda().double()
    d = Q.diagonal().clone()
    U = Q.triu(1)
    g = d + X @ (U + U.T)
    E = (X * (d + g)).sum(1) / 2
    fields = None if case["dtype"] != "fp32" else g.cpu().numpy()
    return dict(fields=fields, energy=E.cpu().numpy())
