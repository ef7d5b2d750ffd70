"""The measured work of this library: what a program has it do through the
public entry points of ``paper_2403_06362_gb300``, over the range of sizes,
seedings, precisions and schedules that the library's own workloads, tests
and benchmark use.

A case is a dict of plain values; ``kind`` names the entry point:

  seed        mc_seed_hash / mc_seed_stride: states only
  draw        mc_lcg_draw on device buffers, fused seeding
  draw_host   mc_lcg_draw_host: results in page-locked host memory
  slab        mc_transport_run, one slab problem
  batched     mc_transport_run, many uneven slab problems in one call
  box         mc_transport_run, two-region multigroup box with a mesh tally
  pulse       mc_transport_run, the time-dependent pulse problem of the
              paper's Section 5, with or without census phases

The seed of ``prepare`` picks the streams (the global hash seed, or X_0 of
the stride baseline) and where the id range starts, so inputs of another seed
are other histories of the same workload.  One library context serves the
whole process, as a program keeps it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2403_06362_gb300 as mc
from paper_2403_06362_gb300 import workloads as W

SEEDINGS = {"hash": W.SEED_HASH, "stride": W.SEED_STRIDE, "hier": W.SEED_HASH_HIER}

# Integer operations one uniform of Eq. (1) takes: 3 for the 64-bit
# multiply-add, 8 to extract, normalise and exponent-insert its 53 bits.
OPS_PER_DRAW = 11
# Operations a flight cannot do without (draws, one logarithm, the geometry
# and the tally contributions), by kind: a count of the method's steps, not of
# instructions.
OPS_PER_FLIGHT = {"slab": 100, "batched": 100, "box": 300, "pulse": 100}
BOX_FLIGHTS = 27.3   # flights per source history of the box workload, children included
PULSE_GROWTH = 0.1   # k - 1 of the pulse problem: its population grows as exp(0.1 t)

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = mc.Context(0)
    return _ctx


def listed():
    return [
        # A handful of streams with every result asked for: launch latency.
        dict(name="draw_small", kind="draw", seeding="hash", streams=4099, draws=16, uniforms=True, digest=True),
        # Seeding a large run's streams by the stride baseline.
        dict(name="seed_stride", kind="seed", seeding="stride", streams=2**26),
        # The random number microbenchmark: seed, 64 draws, final state and digest.
        dict(name="draw_digest", kind="draw", seeding="hash", streams=2**26, draws=64, uniforms=False, digest=True),
        # A program that wants the uniforms themselves in memory.
        dict(name="draw_uniforms", kind="draw", seeding="stride", streams=2**22, draws=64, uniforms=True,
             digest=False),
        # A host program that wants states and digests in its own memory.
        dict(name="draw_host", kind="draw_host", seeding="stride", streams=3_000_001, draws=64),
        # The small slab, run and read back: a whole short calculation.
        dict(name="slab_small", kind="slab", seeding="hash", precision="fp64", schedule="history",
             histories=10_000, L=10.0, sigma_t=1.0, c=0.5, bins=20, batches=10, per_history=True, read=True),
        # The thick, almost purely scattering slab: long, heavy-tailed histories.
        dict(name="slab_long", kind="slab", seeding="hash", precision="fp64", schedule="history",
             histories=1_000_000, L=200.0, sigma_t=1.0, c=0.9999, bins=200, batches=20, per_history=False,
             read=False),
        # A parameter study: 256 uneven slabs in one launch.
        dict(name="slab_batched", kind="batched", seeding="hier", precision="fp32", problems=256,
             max_histories=1_000_000, bins=64),
        # The box with its 64^3 mesh, fp32-guarded flights.
        dict(name="box_fp32", kind="box", seeding="hash", precision="fp32", schedule="history",
             histories=10_000_000, mesh=64),
        # The same in fp64, the parity path, at an odd size.
        dict(name="box_fp64", kind="box", seeding="hash", precision="fp64", schedule="history",
             histories=3_000_001, mesh=64),
        # The paper's experiment at full size.
        dict(name="pulse", kind="pulse", seeding="hier", reps=30, batches=1000, per_batch=1000, phases=0),
        # Census phases with population control, a tenth of the experiment.
        dict(name="pulse_census", kind="pulse", seeding="hier", reps=3, batches=1000, per_batch=1000, phases=20),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["seed", "draw", "draw", "draw_host", "slab", "slab", "batched", "box", "box", "pulse", "pulse"])
    if kind == "seed":
        return dict(kind=kind, seeding=rng.choice(["hash", "stride"]), streams=_log_int(rng, 1_000, 2**26))
    if kind == "draw":
        uniforms = rng.random() < 0.5
        return dict(kind=kind, seeding=rng.choice(["hash", "stride", "hier"]),
                    streams=_log_int(rng, 1_000, 2**22 if uniforms else 2**26),
                    draws=rng.choice([1, 7, 16, 33, 64]), uniforms=uniforms, digest=(not uniforms) or rng.random() < 0.5)
    if kind == "draw_host":
        return dict(kind=kind, seeding=rng.choice(["hash", "stride"]), streams=_log_int(rng, 10_000, 8_000_000),
                    draws=rng.choice([16, 33, 64]))
    if kind == "slab":
        event = rng.random() < 0.25
        long_chains = rng.random() < 0.5
        return dict(kind=kind, seeding=rng.choice(["hash", "stride", "hier"]),
                    precision=rng.choice(["fp64", "fp32"]), schedule="event" if event else "history",
                    histories=_log_int(rng, 1_000, 200_000 if event and long_chains else 1_000_000),
                    L=rng.uniform(20.0, 200.0) if long_chains else rng.uniform(1.0, 50.0),
                    sigma_t=rng.uniform(0.5, 1.0),
                    c=rng.uniform(0.99, 0.9999) if long_chains else rng.uniform(0.1, 0.99),
                    bins=rng.choice([20, 64, 101, 200]), batches=rng.choice([1, 10, 20]),
                    per_history=rng.random() < 0.25, read=rng.random() < 0.25)
    if kind == "batched":
        return dict(kind=kind, seeding=rng.choice(["hier", "stride"]), precision=rng.choice(["fp64", "fp32"]),
                    problems=_log_int(rng, 16, 256), max_histories=_log_int(rng, 3_000, 1_000_000),
                    bins=rng.choice([20, 64, 101]))
    if kind == "box":
        event = rng.random() < 0.25
        return dict(kind=kind, seeding=rng.choice(["hash", "stride", "hier"]),
                    precision=rng.choice(["fp64", "fp32"]), schedule="event" if event else "history",
                    histories=_log_int(rng, 10_000, 3_000_000), mesh=rng.choice([32, 50, 64, 100]))
    phases = rng.choice([0, 0, 2, 10, 20])
    return dict(kind="pulse", seeding=rng.choice(["hier", "hash"] if phases else ["hier", "hash", "stride"]),
                reps=rng.randint(1, 6), batches=_log_int(rng, 10, 1_000), per_batch=_log_int(rng, 100, 1_000),
                phases=phases)


# ----------------------------------------------------------------- preparation

def _streams(case, seed):
    """The stream family of a seed: (global hash seed or X_0, key, first id)."""
    r = np.random.default_rng([seed, 2403])
    if case["seeding"] == "stride":
        return int(r.integers(1, 2**62)) | 1, 0, int(r.integers(0, 2**20))
    return int(r.integers(1, 2**62)), int(r.integers(0, 2**16)), int(r.integers(0, 2**40))


def _problem_seed(case, seed):
    return _streams(case, seed)[0]


def _config(case):
    cfg = mc.mc_run_config()
    cfg.precision = mc.MC_FP32_GUARDED if case.get("precision") == "fp32" else mc.MC_FP64
    cfg.schedule = mc.MC_SCHED_EVENT if case.get("schedule") == "event" else mc.MC_SCHED_HISTORY
    return cfg


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, ctx=_context(), lcg=mc.make_lcg(W.LCG_M, W.LCG_G, W.LCG_C))
    if kind in ("seed", "draw", "draw_host"):
        s, key, begin = _streams(case, seed)
        st.update(seed=s, key=key, begin=begin)
        n = case["streams"]
        if kind == "draw_host":
            st["states"] = torch.zeros(n, dtype=torch.int64).pin_memory()
            st["digest"] = torch.zeros(n, dtype=torch.int64).pin_memory()
        else:
            st["states"] = torch.zeros(n, dtype=torch.int64, device="cuda")
            st["digest"] = torch.zeros(n, dtype=torch.int64, device="cuda") if case.get("digest") else None
            st["u"] = (torch.zeros(case["draws"] * n, dtype=torch.float64, device="cuda")
                       if case.get("uniforms") else None)
        st["spec"] = mc.mc_seed_spec(mode=SEEDINGS[case["seeding"]], reserved=0, seed=s, stride_q=W.STRIDE_Q, key=key)
        return st
    seeding = SEEDINGS[case["seeding"]]
    s = _problem_seed(case, seed)
    st["cfg"] = _config(case)
    if kind == "slab":
        p = [W.slab_problem(case["L"], case["sigma_t"], case["c"], case["histories"], case["bins"], case["batches"],
                            seeding, seed=s, key=_streams(case, seed)[1])]
    elif kind == "batched":
        p = W.slab_batched(seeding, n_problems=case["problems"], n_bins=case["bins"],
                           max_histories=case["max_histories"])
        for q in p:
            q["seed"] = s
    if kind in ("slab", "batched"):
        st["problems"] = mc.problem_array([W.to_mc_problem(q, mc) for q in p])
        st["tally"] = mc.Tally(W.tally_slots(p), len(p), n_histories=case["histories"] if case.get("per_history") else 0)
        return st
    if kind == "box":
        b = W.box_problem(n_histories=case["histories"], seeding=seeding, mesh=case["mesh"], seed=s)
        prob, st["spec"] = W.to_mc_box(b, mc)
        slots = W.box_tally_slots(b)
    else:
        a = W.azurv1(seeding=seeding, n_reps=case["reps"], n_batches=case["batches"], per_batch=case["per_batch"],
                     seed=s, n_census=case["phases"])
        prob, st["spec"] = W.to_mc_pulse(a, mc)
        slots = W.azurv1_tally_slots(a)
    st["problems"] = mc.problem_array([prob])
    st["tally"] = mc.Tally(slots, 1)
    return st


# ------------------------------------------------------------------------ runs

def run(st):
    case, ctx, lcg = st["case"], st["ctx"], st["lcg"]
    kind = case["kind"]
    if kind == "seed":
        if case["seeding"] == "stride":
            mc.mc_seed_stride(ctx, lcg, st["seed"], W.STRIDE_Q, st["begin"], case["streams"], st["states"])
        else:
            mc.mc_seed_hash(ctx, lcg, st["seed"], st["begin"], case["streams"], st["states"])
        return {"states": st["states"]}
    if kind == "draw":
        mc.mc_lcg_draw(ctx, lcg, st["spec"], st["begin"], st["states"], case["streams"], case["draws"], st["u"],
                       st["digest"])
        return {k: st[k] for k in ("states", "u", "digest") if st[k] is not None}
    if kind == "draw_host":
        mc.mc_lcg_draw_host(ctx, lcg, st["spec"], st["begin"], st["states"], case["streams"], case["draws"],
                            st["digest"])
        return {"states": st["states"], "digest": st["digest"]}
    t = st["tally"]
    mc.mc_transport_run(ctx, lcg, st["problems"], st["cfg"], t.c)
    out = {"bins": t.bins, "counts": t.counts}
    if t.hist_state is not None:
        out["hist_state"], out["hist_draws"] = t.hist_state, t.hist_draws
    if case.get("read"):
        r = mc.mc_tally_read(ctx, st["problems"], 0, t.c)
        out["flux"], out["rel_err"], out["batch"] = r.flux, r.rel_err, r.batch
    return out


# ------------------------------------------------------------------------ work

def _slab_flights(L, sigma_t, c):
    """Expected flights per history of a uniform isotropic source: the leak
    probability per flight is the first-flight escape of a thin slab and the
    diffusion decay rate (pi / (tau + 1.42))^2 / 3 of a thick one."""
    tau = L * sigma_t
    escape = min(1.0, (1.0 - 2.0 * math.exp(-tau) / (tau + 2.0)) / (2.0 * tau))
    leak = min(escape, (math.pi / (tau + 1.42)) ** 2 / 3.0)
    return 1.0 / (1.0 - c * (1.0 - leak))


def work(case):
    kind = case["kind"]
    if kind == "seed":
        return {"bytes": 8 * case["streams"], "flops": OPS_PER_DRAW * case["streams"]}
    if kind in ("draw", "draw_host"):
        n, d = case["streams"], case["draws"]
        per_stream = 8 + (8 if kind == "draw_host" or case["digest"] else 0) + (8 * d if case.get("uniforms") else 0)
        return {"bytes": n * per_stream, "flops": OPS_PER_DRAW * n * d}
    if kind == "slab":
        flights = case["histories"] * _slab_flights(case["L"], case["sigma_t"], case["c"])
        out = 8 * case["bins"] * case["batches"] + (16 * case["histories"] if case["per_history"] else 0)
    elif kind == "batched":
        p = W.slab_batched(SEEDINGS[case["seeding"]], n_problems=case["problems"], n_bins=case["bins"],
                           max_histories=case["max_histories"])
        flights = sum(q["n_histories"] * _slab_flights(q["L"], q["sigma_t"], q["c"]) for q in p)
        out = 8 * case["bins"] * case["problems"]
    elif kind == "box":
        flights = case["histories"] * BOX_FLIGHTS
        out = 8 * case["mesh"] ** 3
    else:
        sources = case["reps"] * case["batches"] * case["per_batch"]
        if case["phases"] >= 2:  # control holds the population; a phase starts every particle's flight anew
            t_phase = 20.0 / case["phases"]
            flights = sources * case["phases"] * (1.0 + math.expm1(PULSE_GROWTH * t_phase) / PULSE_GROWTH)
        else:
            flights = sources * (1.0 + math.expm1(PULSE_GROWTH * 20.0) / PULSE_GROWTH)
        out = 8 * 20 * case["reps"] * case["batches"]
    return {"bytes": out + 8 * mc.MC_NCOUNT, "flops": OPS_PER_FLIGHT[kind] * flights}


# ----------------------------------------------------------------- 64-bit truth

_MURMUR = 0xC6A4A7935BD1E995


def _i64(v):
    """The two's-complement int64 of a 64-bit word."""
    v &= 2**64 - 1
    return v - 2**64 if v >= 2**63 else v


def _lsr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _mix(x):
    t = x * _i64(_MURMUR)
    return t ^ _lsr(t, 47)


def _hash_int(k, s):
    m64 = 2**64 - 1

    def mix(x):
        t = (x * _MURMUR) & m64
        return t ^ (t >> 47)
    return mix(mix(s ^ ((8 * _MURMUR) & m64)) ^ ((mix(k) * _MURMUR) & m64))


def _hash(k, s):
    """hash(k, s) of Listing 1 for an int64 tensor of keys and a 64-bit seed."""
    m64 = 2**64 - 1
    t = ((s ^ ((8 * _MURMUR) & m64)) * _MURMUR) & m64
    return _mix(_mix(k) * _i64(_MURMUR) ^ _i64(t ^ (t >> 47)))


_MASK63 = 2**63 - 1


def _seeds(seeding, s, key, begin, n):
    """States of units begin .. begin + n - 1 (Eqs. 2-4), int64 tensor."""
    ids = torch.arange(n, dtype=torch.int64, device="cuda") + begin
    if seeding != "stride":
        return _hash(ids, _hash_int(key, s) if seeding == "hier" else s) & _MASK63
    x = torch.full((n,), _i64(s), dtype=torch.int64, device="cuda")
    a, b, m64 = W.LCG_G, W.LCG_C, 2**64 - 1
    steps = ids * W.STRIDE_Q
    for j in range(64):  # the map of 2^j steps, applied where bit j of the step count is set
        if (begin + n) * W.STRIDE_Q >> j == 0:
            break
        x = torch.where((steps >> j) & 1 == 1, x * _i64(a) + _i64(b), x)
        a, b = (a * a) & m64, (a * b + b) & m64
    return x & _MASK63


def _step(x):
    return (x * _i64(W.LCG_G) + W.LCG_C) & _MASK63


def _uniform(x):
    return (x >> 10).double() * 2.0**-53


def exact(case, seed):
    kind = case["kind"]
    if kind == "slab":
        return _exact_slab(case, seed)
    if kind not in ("seed", "draw", "draw_host"):
        return None  # every output is a whole number
    s, key, begin = _streams(case, seed)
    x = _seeds(case["seeding"], s, key, begin, case["streams"])
    if kind == "seed":
        return {"states": x}
    dg = torch.zeros_like(x)
    u = torch.empty(case["draws"], case["streams"], dtype=torch.float64, device="cuda") if case.get("uniforms") else None
    for j in range(case["draws"]):
        x = _step(x)
        v = _uniform(x)
        dg += v.view(torch.int64)
        if u is not None:
            u[j] = v
    out = {"states": x}
    if u is not None:
        out["u"] = u.reshape(-1)
    if kind == "draw_host" or case.get("digest"):
        out["digest"] = dg
    return out


def _exact_slab(case, seed):
    """The flux of a slab read back, by plain fp64 steps over all histories at
    once; None where that takes too many steps or nothing is read back."""
    n, nb, nbat = case["histories"], case["bins"], case["batches"]
    if not case["read"] or _slab_flights(case["L"], case["sigma_t"], case["c"]) > 40.0 or n > 200_000:
        return None
    L, st, c = case["L"], case["sigma_t"], case["c"]
    s, key, _ = _streams(case, seed)
    r = _seeds(case["seeding"], s, key, 0, n)
    ids = torch.arange(n, dtype=torch.int64, device="cuda")
    row = ids * nbat // n * nb
    lo = torch.arange(nb, dtype=torch.float64, device="cuda") * (L / nb)
    hi = torch.cat([lo[1:], torch.tensor([L], dtype=torch.float64, device="cuda")])
    bins = torch.zeros(nbat * nb, dtype=torch.float64, device="cuda")
    r = _step(r)
    x = L * _uniform(r)
    r = _step(r)
    mu = 2.0 * _uniform(r) - 1.0
    while r.numel():
        r = _step(r)
        d = -torch.log(1.0 - _uniform(r)) / st
        xn = x + d * mu
        out = ((mu > 0) & (xn >= L)) | ((mu < 0) & (xn <= 0))
        a, b = torch.minimum(x, xn).clamp(min=0.0), torch.maximum(x, xn).clamp(max=L)
        w = 1.0 / mu.abs()
        for j in range(nb):
            bins.index_add_(0, row + j, (torch.minimum(b, hi[j]) - torch.maximum(a, lo[j])).clamp(min=0.0) * w)
        keep = ~out
        r, x, row = r[keep], xn[keep], row[keep]
        r = _step(r)
        keep = _uniform(r) >= 1.0 - c
        r, x, row = r[keep], x[keep], row[keep]
        r = _step(r)
        mu = 2.0 * _uniform(r) - 1.0
    v = bins.reshape(nbat, nb).cpu().numpy()
    h = L / nb
    k = np.arange(nbat + 1)
    first = -(-k * n // nbat)
    batch = v / (np.diff(first)[:, None] * h)
    flux = v.sum(axis=0) / (n * h)
    rel = np.zeros(nb)
    if nbat >= 2:
        rel = np.where(flux != 0, batch.std(axis=0, ddof=1) / math.sqrt(nbat) / np.where(flux != 0, flux, 1.0), 0.0)
    return {"bins": None, "counts": None, "hist_state": None, "hist_draws": None, "flux": flux, "rel_err": rel,
            "batch": batch}
