"""The work that programs have this library do, as cases to be timed.

Every case goes through the Python binding's public calls: whole runs of
Algorithm 1 (smc.run), many runs together (smc.run_batch), a burst of requests to
the continuous-batching server (smc.Server), the standalone resampling step
(smc.resample) and the particle duplication (smc.gather).  Sizes come from the
repository's benchmark workloads and tests, beside odd ones of the same ranges.

A case's "seed" argument gives the data (observations, tree, log-weights) and the
run's Philox key; its sizes and options are the case's own.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import inputs
from paper_2112_00364_gb300 import smc

# Elementary operations of one particle-step that the model's own formulas need
# (an elementary function counted as 10, a hidden-lineage event of the tree
# models at its usual frequency), the weight, its running sum and the search
# included.
STEP_FLOPS = {"lg": 60, "crbd": 80, "rateshift": 130, "crbd_ds": 140, "seir": 900}
RATE_STACK = 20
N_REAL = {"lg": 1, "crbd": 2, "rateshift": 2, "crbd_ds": 4, "seir": 6}
N_INT = {"lg": 1, "crbd": 1, "rateshift": 2, "crbd_ds": 1, "seir": 10}


def listed():
    return [
        # the smallest calls: the textbook state-space model at its usual size, and a
        # small phylogeny with single-precision particles; results on the host, as a
        # script reads them
        {"name": "lg_1k", "do": "run", "kind": "lg", "N": 1024, "length": 50, "precision": "fp64",
         "where": "host"},
        {"name": "crbd_512_fp32", "do": "run", "kind": "crbd", "N": 512, "length": 32,
         "precision": "fp32", "where": "host"},
        # an ordinary filtering run of odd size that keeps its whole genealogy (for
        # smoothing): short segments one after another
        {"name": "lg_23k_genealogy", "do": "run", "kind": "lg", "N": 23171, "length": 118,
         "precision": "fp64", "where": "device", "record_all": True},
        # the birth-death model on a 64-tip tree, the default benchmark workload
        {"name": "crbd_64k", "do": "run", "kind": "crbd", "N": 65536, "length": 64,
         "precision": "fp64", "where": "device"},
        # static delayed sampling with ESS-triggered resampling on a 128-tip tree
        {"name": "crbd_ds_100k_ess", "do": "run", "kind": "crbd_ds", "N": 100000, "length": 128,
         "precision": "fp64", "where": "device", "ess": 0.5},
        # half a year of epidemic reports: thirteen binomial draws a particle and day
        {"name": "seir_64k", "do": "run", "kind": "seir", "N": 65536, "length": 182,
         "precision": "fp64", "where": "device"},
        # a large population with a stack that crosses checkpoints
        {"name": "rateshift_1m_fp32", "do": "run", "kind": "rateshift", "N": 1 << 20, "length": 256,
         "precision": "fp32", "where": "device"},
        # many uneven runs of two models in one call
        {"name": "batch_512_fp32", "do": "batch", "runs": 512, "specs": 4, "precision": "fp32"},
        # a burst of requests to the server, from the first submission to the last result
        {"name": "serve_96_fp32", "do": "serve", "runs": 96, "specs": 5, "precision": "fp32"},
        # the resampling step of a program with particles of its own: a large population,
        # and a small odd one with the duplication of a three-field state
        {"name": "resample_16m", "do": "resample", "N": 1 << 24, "scale": 2.0, "dead": 0.0},
        {"name": "resample_copy_100k", "do": "resample_copy", "N": 100003, "scale": 3.0, "dead": 0.2,
         "rows": 3, "bytes": 8, "stack": False},
        # duplication of stack-bearing single-precision states, rows above the stack
        # pointer left alone
        {"name": "copy_stack_4m_fp32", "do": "copy", "N": (1 << 22) + 5, "scale": 2.0, "dead": 0.0,
         "rows": 12, "bytes": 4, "stack": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["lg", "crbd", "crbd_ds", "rateshift", "seir", "batch", "serve", "resample",
                     "resample_copy", "copy"])
    if do == "batch":
        return {"do": do, "runs": _log_int(rng, 8, 256), "specs": rng.randrange(1, 1000),
                "precision": rng.choice(["fp32", "fp64"])}
    if do == "serve":
        return {"do": do, "runs": _log_int(rng, 8, 192), "specs": rng.randrange(1, 1000),
                "precision": "fp32"}
    if do in ("resample", "resample_copy", "copy"):
        lo, hi = {"resample": (300, 1 << 24), "resample_copy": (300, 1 << 22),
                  "copy": (200000, 1 << 22)}[do]
        case = {"do": do, "N": _log_int(rng, lo, hi),
                "scale": round(rng.uniform(0.5, 4.0), 2), "dead": rng.choice([0.0, 0.2])}
        if do != "resample":
            case.update(rows=rng.randrange(1, 13), bytes=rng.choice([4, 8]),
                        stack=rng.choice([False, True]))
        return case
    hi = {"lg": 1 << 19, "crbd": 1 << 18, "crbd_ds": 1 << 17, "rateshift": 1 << 19, "seir": 1 << 16}
    length = {"lg": (20, 500), "crbd": (16, 256), "crbd_ds": (16, 128), "rateshift": (16, 256),
              "seir": (28, 182)}
    case = {"do": "run", "kind": do, "N": _log_int(rng, 100, hi[do]),
            "length": _log_int(rng, *length[do]), "precision": rng.choice(["fp64", "fp32"]),
            "where": rng.choice(["device", "device", "host"])}
    if rng.random() < 0.25:
        case["ess"] = 0.5
    return case


# ---- data ----

def _model(kind, length, seed):
    """A registered model with data of its own: observations (lg, seir) or a tree."""
    if kind == "lg":
        return smc.Model("lg", obs=inputs.lg_observations(length, seed=seed))
    if kind == "seir":
        return smc.Model("seir", obs=inputs.seir_observations(length, seed=seed))
    tree = inputs.yule_tree(length, seed=seed)
    if kind == "rateshift":
        # one capacity for every tree, as a program that has many would choose it
        return smc.Model("rateshift", tree=tree, sigma=0.3, lam_stack_cap=RATE_STACK)
    return smc.Model(kind, tree=tree)


def _logw(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.randn(case["N"], generator=gen, dtype=torch.float64, device="cuda") * case["scale"]
    if case["dead"]:
        dead = torch.rand(case["N"], generator=gen, device="cuda") < case["dead"]
        dead[0] = False  # never a population without a survivor
        x[dead] = -math.inf
    return x


def _uniform(seed):
    return float(np.random.Generator(np.random.PCG64(seed)).uniform(0.05, 0.95))


def _population(case, seed):
    """A state of `rows` fields and its stack pointers (None: every row is copied)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    dt = torch.float32 if case["bytes"] == 4 else torch.float64
    src = torch.randn(case["rows"], case["N"], generator=gen, dtype=dt, device="cuda")
    sp = None
    if case["stack"]:
        sp = torch.randint(0, case["rows"] + 1, (case["N"],), generator=gen, dtype=torch.int32,
                           device="cuda")
    return src, sp


def prepare(case, seed):
    do, seed = case["do"], int(seed)
    if do == "run":
        m = _model(case["kind"], case["length"], seed)
        state = {"do": do, "case": case, "model": m, "seed": seed}
        if case["where"] == "device":
            n, rows = case["N"], m.n_segments - 1 if case.get("record_all") else 1
            f8 = dict(dtype=torch.float64, device="cuda")
            i4 = dict(dtype=torch.int32, device="cuda")
            out = {"log_z": torch.zeros(1, **f8), "final_logw": torch.zeros(n, **f8),
                   "ancestors": torch.zeros(rows, n, **i4),
                   "real_fields": torch.zeros(m.n_real, n, **f8),
                   "int_fields": torch.zeros(m.n_int, n, **i4), "resampled": torch.zeros(rows, **i4)}
            if m.stack_cap:
                out["stack"] = torch.zeros(m.stack_cap, n, **f8)
            state["out"] = out
        return state
    if do in ("batch", "serve"):
        specs = inputs.batch_specs(case["runs"], seed=case["specs"])
        models, runs = [], []
        total = sum(s.n_particles for s in specs)
        reals = sum(s.n_particles * N_REAL[s.kind] for s in specs)
        f8 = dict(dtype=torch.float64, device="cuda")
        i4 = dict(dtype=torch.int32, device="cuda")
        # one allocation per kind of output, a slice of it for each run
        packed = {"log_z": torch.zeros(len(specs), **f8), "final_logw": torch.zeros(total, **f8),
                  "ancestors": torch.zeros(total, **i4), "real_fields": torch.zeros(reals, **f8),
                  "int_fields": torch.zeros(total, **i4), "resampled": torch.zeros(len(specs), **i4)}
        at = at_real = 0
        for q, s in enumerate(specs):
            n, nr = s.n_particles, N_REAL[s.kind]
            models.append(_model(s.kind, s.T or s.tips, seed * 1009 + q))
            runs.append({"N": n, "seed": seed, "run_id": q, "outputs": {
                "log_z": packed["log_z"][q:q + 1], "final_logw": packed["final_logw"][at:at + n],
                "ancestors": packed["ancestors"][at:at + n].view(1, n),
                "real_fields": packed["real_fields"][at_real:at_real + nr * n].view(nr, n),
                "int_fields": packed["int_fields"][at:at + n].view(1, n),
                "resampled": packed["resampled"][q:q + 1]}})
            at, at_real = at + n, at_real + nr * n
        state = {"do": do, "case": case, "models": models, "runs": runs, "packed": packed}
        if do == "serve":
            state["server"] = smc.Server(16 << 30, precision=case["precision"])
        return state
    state = {"do": do, "u": _uniform(seed)}
    lw = _logw(case, seed)
    n = case["N"]
    state["anc"] = torch.empty(n, dtype=torch.int32, device="cuda")
    if do == "copy":
        # the ancestors of a systematic resampling, formed with plain torch
        w = torch.exp(lw - lw.max())
        q = torch.cumsum(w, 0)
        q = q * (n / q[-1])
        at = torch.arange(n, dtype=torch.float64, device="cuda") + state["u"]
        state["anc"].copy_(torch.searchsorted(q, at, right=True).clamp_(max=n - 1))
    else:
        state["logw"] = lw
        state["out3"] = torch.empty(3, dtype=torch.float64, device="cuda")
        state["near"] = torch.empty(1, dtype=torch.int64, device="cuda")
        state["work"] = torch.empty(smc.resample_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    if do != "resample":
        state["src"], state["sp"] = _population(case, seed)
        state["dst"] = torch.zeros_like(state["src"])
    return state


# ---- one pass ----

COUNTERS = ("status", "n_segments", "n_resamples", "n_near_boundary", "n_overflow", "n_limit",
            "n_ess_near", "n_draws", "n_blocks")
OUTPUTS = ("log_z", "final_logw", "ancestors", "real_fields", "int_fields", "stack", "resampled")


def run(state):
    do = state["do"]
    if do == "run":
        case = state["case"]
        res = smc.run(state["model"], case["N"], state["seed"], precision=case["precision"],
                      where=case["where"], record_all_ancestors=bool(case.get("record_all")),
                      ess_threshold=case.get("ess", 0.0), outputs=state.get("out"))
        return {k: res[k] for k in OUTPUTS + COUNTERS if k in res}
    if do == "batch":
        res = smc.run_batch(state["models"], state["runs"], precision=state["case"]["precision"],
                            where="device")
    elif do == "serve":
        srv = state["server"]
        tickets = [srv.submit(m, r["N"], r["seed"], run_id=r["run_id"], where="device",
                              outputs=r["outputs"])
                   for m, r in zip(state["models"], state["runs"])]
        res = [srv.wait(t) for t in tickets]
    else:
        if do != "copy":
            smc.resample(state["logw"], state["u"], ancestors=state["anc"], out3=state["out3"],
                         n_near=state["near"], workspace=state["work"])
        out = {}
        if do != "copy":
            out = {"ancestors": state["anc"], "out3": state["out3"], "near": state["near"]}
        if do != "resample":
            out["state"] = smc.gather(state["src"], state["dst"], state["anc"], sp=state["sp"])
        return out
    return {**state["packed"],
            "counters": np.array([[r[k] for k in COUNTERS] for r in res], dtype=np.int64)}


# ---- what a pass cannot do without ----

def _run_work(kind, n, length, stack_rows=0, rows=1):
    segments = length if kind in ("lg", "seir") else 2 * length - 1
    # the data in, the final states, log-weights and ancestor rows out
    data = 8 * length if kind in ("lg", "seir") else 32 * segments
    bytes_ = data + n * (8 + 4 * rows + 8 * (N_REAL[kind] + stack_rows) + 4 * N_INT[kind])
    return bytes_, n * segments * STEP_FLOPS[kind]


def work(case):
    do = case["do"]
    if do == "run":
        rows = case["length"] - 1 if case.get("record_all") and case["kind"] == "lg" else 1
        b, f = _run_work(case["kind"], case["N"], case["length"], rows=rows)
        return {"bytes": b, "flops": f}
    if do in ("batch", "serve"):
        both = [_run_work(s.kind, s.n_particles, s.T or s.tips)
                for s in inputs.batch_specs(case["runs"], seed=case["specs"])]
        return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}
    n, b, f = case["N"], 0, 0
    if do != "copy":  # log-weight in, ancestor out; an exponential, a sum and a comparison
        b, f = b + 12 * n, f + 13 * n
    if do != "resample":
        rows = case["rows"] / 2 if case["stack"] else case["rows"]
        b += n * (4 + (4 if case["stack"] else 0) + 2 * case["bytes"] * rows)
    return {"bytes": b, "flops": f}


# ---- the same in plain numpy, 64 bits ----

def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 over arrays of counters (uint64 arrays of 32-bit words)."""
    m32 = np.uint64(0xFFFFFFFF)
    s32 = np.uint64(32)
    c = [np.asarray(x, dtype=np.uint64) for x in (c0, c1, c2, c3)]
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    for r in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> s32) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> s32) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _unit(lo, hi):
    bits = (np.asarray(hi, dtype=np.uint64) << np.uint64(32)) | np.asarray(lo, dtype=np.uint64)
    return ((bits >> np.uint64(11)) | np.uint64(1)).astype(np.float64) * 2.0 ** -53


def _exact_lg(case, seed):
    n, T = case["N"], case["length"]
    y = inputs.lg_observations(T, seed=int(seed))
    i = np.arange(n, dtype=np.uint64)
    zero = np.zeros(n, dtype=np.uint64)
    key = int(seed)

    def normal(k, d):
        w = _philox(i, zero + np.uint64(k), zero + np.uint64(d), zero, key)
        return np.sqrt(-2.0 * np.log(_unit(w[0], w[1]))) * np.cos(2.0 * np.pi * _unit(w[2], w[3]))

    x, log_z, tau = normal(0, 0), 0.0, case.get("ess", 0.0)
    acc = np.zeros(n)
    for k in range(T):
        x = 0.9 * x + normal(k, 1 if k == 0 else 0)
        lw = acc - 0.5 * ((y[k] - x) / 0.5) ** 2 - math.log(0.5) - 0.5 * math.log(2.0 * math.pi)
        m = lw.max()
        w = np.exp(lw - m)
        cum = np.cumsum(w.astype(np.longdouble))
        total = float(cum[-1])
        inc = m + math.log(total) - math.log(n)
        resample = tau == 0.0 or total * total / float(np.sum(w * w)) < tau * n
        if k == T - 1 or resample:
            log_z += inc
        if k == T - 1:
            return {"log_z": np.array([log_z]), "final_logw": lw, "real_fields": x[None, :].copy()}
        acc = lw
        if resample:
            u = _unit(*_philox(np.uint64(0), np.uint64(k), np.uint64(0), np.uint64(1), key)[:2])
            q = cum * (np.longdouble(n) / cum[-1])
            a = np.searchsorted(q, np.arange(n, dtype=np.longdouble) + np.longdouble(u), side="right")
            x, acc = x[np.minimum(a, n - 1)], np.zeros(n)


def exact(case, seed):
    do = case["do"]
    if do == "run":
        # The tree models and the epidemic model draw a varying number of variates per
        # particle from recursions: a plain 64-bit restatement takes minutes.  With
        # single-precision particles other ancestors are drawn than in 64 bits, so no
        # particle has a 64-bit value of its own.
        small = case["N"] * case["length"] <= 1 << 23
        return _exact_lg(case, seed) if case["kind"] == "lg" and case["precision"] == "fp64" and small else None
    if do in ("batch", "serve"):
        return None
    state = prepare(case, seed)
    out = {}
    if do != "copy":
        lw = state["logw"].cpu().numpy()
        top = math.ceil(lw.max() / math.log(2.0)) * math.log(2.0)  # the power-of-two reference
        w = np.exp(lw - top)
        cum = np.cumsum(w.astype(np.longdouble))
        s = float(cum[-1])
        out["out3"] = np.array([top, s, top + math.log(s) - math.log(case["N"])])
        q = cum * (np.longdouble(case["N"]) / cum[-1])
        at = np.arange(case["N"], dtype=np.longdouble) + np.longdouble(state["u"])
        anc = np.minimum(np.searchsorted(q, at, side="right"), case["N"] - 1)
    else:
        anc = state["anc"].cpu().numpy()
    if do != "resample":
        src = state["src"].cpu().numpy()
        dst = src[:, anc].astype(np.float64)
        if state["sp"] is not None:  # rows from the stack pointer on stay as they were
            sp = state["sp"].cpu().numpy()[anc]
            dst[np.arange(case["rows"])[:, None] >= sp[None, :]] = 0.0
        out["state"] = dst
    return out
