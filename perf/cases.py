"""Workloads of the scheduler library: what a program that schedules with it has it do.

Every case goes through the package's public calls (``paper_2405_06856_gb300.aladdin``):

* ``heartbeat``: the workers' new state and the waiting requests arrive on the device, one
  ``aladdin_cluster_load_score`` call loads the state and scores every (request, worker) pair;
* ``score``: ``aladdin_score`` against a state that was loaded before;
* ``round``: the workers' new state is loaded and the waiting requests are placed greedily
  (``aladdin_place_round``); a case may then score more requests against the open round;
* ``simulate``: ``aladdin_simulate`` of a request trace on a fixed fleet (host arrays in, nine numbers
  out);
* ``search``: ``aladdin_min_workers``, the smallest fleet per worker size that serves a trace, then a
  simulation of the chosen fleet for the latencies it realizes.

Lengths, rates, coefficients and sizes are those of the package's workload recipe: lognormal prompt and
output lengths, generated tokens uniform below the prediction, waits uniform in [0, 100) ms, 1/2/4/8-GPU
workers with KV capacity proportional to the GPUs and latency coefficients x 1/sqrt(GPUs).
"""
import math

import numpy as np
import torch

from paper_2405_06856_gb300 import aladdin as A

BASE = dict(k1=0.001, c1=10.0, k2=2e-4, c2=0.05, c3=8.0, h=1, j=0, T_pre=1000.0, T_dec=50.0,
            gamma=0.5, theta=1.0, K=8192)
IN_LAW = (512.0, 0.8, 16, 2048)
OUT_LAW = (256.0, 0.9, 8, 1024)
HEAVY_OUT = (256.0, 1.2, 8, 4096)
GPU_MIX = (1, 2, 4, 8)

MODES = {"exact": A.MODE_EXACT, "approx": A.MODE_APPROX}
PHASES = {"mixed": A.PHASE_MIXED, "decode": A.PHASE_DECODE}
POLICIES = {"bestfit": A.POLICY_BESTFIT, "jsq": A.POLICY_JSQ, "po2": A.POLICY_PO2}


def _fleet(name, call, workers, per_worker, cands, kv, slots, **more):
    """A case over a fixed fleet. ``spread``: a worker holds 0..per_worker requests, not exactly that many;
    ``gpu_mix``: workers of 1/2/4/8 GPUs in turn; ``heavy``: the heavy-tailed output law; ``history``: the
    requests' decode time so far is given; ``outputs``: f(lags), m(argins), a(rgbest); ``memory``: where the
    caller's arrays lie."""
    case = dict(call=call, workers=workers, per_worker=per_worker, cands=cands, kv=kv, slots=slots,
                spread=False, gpu_mix=False, heavy=False, history=False, outputs="fma",
                memory="device", mode="exact", phase="mixed", policy="bestfit", groups=1,
                T_pre=1000.0, T_dec=50.0, theta=1.0, then_score=0)
    case.update(more)
    if name:
        case["name"] = name
    return case


def _trace(name, call, requests, rate, workers, kv, slots, **more):
    """A case over a request trace: ``workers`` is the fleet (simulate) or the search bound (search)."""
    case = dict(call=call, requests=requests, rate=rate, workers=workers, kv=kv, slots=slots, gpus=1,
                mode="exact", phase="mixed", policy="bestfit", groups=1, T_pre=1000.0, T_dec=50.0,
                theta=1.0)
    case.update(more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # The smallest deployment: one heartbeat of a 16-worker fleet with 64 waiting requests.
        _fleet("heartbeat_16", "heartbeat", 16, 24, 64, 16384, 64, T_pre=60.0, T_dec=30.0, spread=True),
        # An engine that keeps its arrays in page-locked host memory and reads every result there.
        _fleet("score_256_pinned", "score", 256, 64, 2048, 65536, 128, memory="pinned"),
        # The package's benchmark: one heartbeat of 4,096 workers with 32,768 waiting requests.
        _fleet("heartbeat_4096", "heartbeat", 4096, 128, 32768, 131072, 256, heavy=True),
        # A dispatcher that wants the chosen worker only, on a fleet near its limits (every constraint
        # binds somewhere) whose requests carry their decode history.
        _fleet("argbest_4096", "score", 4096, 128, 32768, 90000, 256, heavy=True, history=True,
               outputs="a", T_pre=95.0, T_dec=30.0),
        # The largest fleet: workers of 1/2/4/8 GPUs, 256 requests each, 1,024 slots.
        _fleet("score_16384", "score", 16384, 256, 32768, 131072, 1024, heavy=True, gpu_mix=True),
        # An odd fleet at odd load under the approximate constraints of the placement program.
        _fleet("score_1001_approx", "score", 1001, 96, 5003, 65536, 256, spread=True, history=True,
               mode="approx", theta=0.9),
        # A small scheduler that hands over plain host arrays: place 96 requests on 33 workers.
        _fleet("round_33_host", "round", 33, 24, 96, 32768, 128, spread=True, memory="host", then_score=32),
        # One greedy round of 2,048 requests on 256 workers, then 256 more scored against the open round.
        _fleet("round_256", "round", 256, 64, 2048, 57344, 128, then_score=256),
        # One of ten heartbeats of the largest workload: 13,107 arrivals on 16,384 mixed workers.
        _fleet("round_16384", "round", 16384, 256, 13107, 131072, 1024, heavy=True, gpu_mix=True,
               then_score=64),
        # Distributed scheduling: 31 independent groups share one round.
        _fleet("round_4096_groups", "round", 4096, 128, 8192, 131072, 512, heavy=True, groups=31, then_score=64),
        # Capacity planning: simulate a day compressed to seconds on a fixed fleet.
        _trace("simulate_128", "simulate", 8000, 1250.0, 128, 65536, 512),
        # Capacity planning: the smallest fleet per worker size for a short trace.
        _trace("search_4_sizes", "search", 1500, 400.0, 256, 65536, 1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _slots_for(kv, gpus):
    """Slots that no worker outgrows: its KV capacity in requests of about 350 tokens."""
    need = kv * gpus / 350.0
    return min(1024, 1 << max(5, math.ceil(math.log2(need))))


def draw(rng):
    call = rng.choice(["heartbeat", "score", "score", "round", "round", "simulate", "search"])
    theta = rng.choice([1.0, 1.0, 0.9])
    phase = rng.choice(["mixed", "mixed", "mixed", "decode"])
    if call == "simulate":
        rate = rng.uniform(300.0, 1500.0)
        return _trace("", call, _log_int(rng, 500, 8000), rate, int(rate * rng.uniform(0.08, 0.16)) + 4,
                      65536, 512, phase=phase, theta=theta, policy=rng.choice(["bestfit", "bestfit", "jsq", "po2"]),
                      groups=rng.choice([1, 1, 1, 3]))
    if call == "search":
        return _trace("", call, _log_int(rng, 300, 1500), rng.uniform(150.0, 400.0), 256, 65536, 1024,
                      phase=phase, theta=theta)
    gpu_mix = rng.random() < 0.3
    if call == "round":
        # a chain of placements: the fleet's size and the arrivals bound it, never both at their largest
        workers = _log_int(rng, 16, 16384)
        cands = _log_int(rng, 32, 8192)
        kv = rng.choice([65536, 131072])
        per_worker = rng.randint(8, 64 if kv == 65536 else 128)
        policy = rng.choice(["bestfit", "bestfit", "bestfit", "jsq", "po2"])
        if policy != "bestfit":  # no feasibility test: leave the slots room for what they are dealt
            workers = min(workers, 12000)
            cands = min(cands, 64 * workers)
        return _fleet("", call, workers, per_worker, cands, kv, _slots_for(kv, 8 if gpu_mix else 1) if policy == "bestfit" else 512,
                      spread=rng.random() < 0.5, gpu_mix=gpu_mix, heavy=rng.random() < 0.5, history=rng.random() < 0.3,
                      memory=rng.choice(["device", "device", "pinned", "host"]), phase=phase, policy=policy,
                      groups=rng.choice([1, 1, 1, 7]) if workers >= 64 else 1, theta=theta,
                      then_score=rng.choice([0, 33, 128]))
    workers = _log_int(rng, 8, 16384)
    cands = _log_int(rng, 32, 32768)
    per_worker = rng.randint(8, 256)
    mode = rng.choice(["exact", "exact", "approx"])
    return _fleet("", call, workers, per_worker, cands, rng.choice([65536, 90000, 131072]),
                  1 << max(5, math.ceil(math.log2(per_worker + 1))), spread=rng.random() < 0.5, gpu_mix=gpu_mix,
                  heavy=rng.random() < 0.5, history=rng.random() < 0.5, outputs=rng.choice(["fma", "fma", "fa", "a", "m"]),
                  memory=rng.choice(["device", "device", "device", "pinned"]) if workers * cands <= 1 << 22 else "device",
                  mode=mode, phase=phase, T_pre=rng.choice([1000.0, 95.0]), T_dec=rng.choice([50.0, 30.0]), theta=theta)


# ---------------------------------------------------------------------------
# Inputs, from the seed alone.

def _params(case):
    return dict(BASE, T_pre=case["T_pre"], T_dec=case["T_dec"], theta=case["theta"], mode=MODES[case["mode"]],
                phase=PHASES[case["phase"]], policy=POLICIES[case["policy"]], groups=case["groups"], seed=12345)


def _lengths(gen, n, law):
    mean, sigma, lo, hi = law
    x = torch.empty(n, dtype=torch.float64, device="cuda").normal_(generator=gen)
    x = torch.exp(math.log(mean) - 0.5 * sigma * sigma + sigma * x)
    return x.round_().clamp_(lo, hi).to(torch.int32)


def _sizes(case):
    """GPUs, KV capacity and latency scale of every worker."""
    W = case["workers"]
    gpus = np.array([GPU_MIX[i % 4] if case["gpu_mix"] else 1 for i in range(W)], np.int32)
    scale = (1.0 / np.sqrt(gpus.astype(np.float64))).astype(np.float32)
    return gpus, gpus.astype(np.int64) * case["kv"], scale


def _requests(case, seed):
    """The workers' ongoing requests (CSR) and the waiting requests, on the device."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    W, out_law = case["workers"], HEAVY_OUT if case["heavy"] else OUT_LAW

    def uniform(n):
        return torch.empty(n, dtype=torch.float64, device="cuda").uniform_(generator=gen)

    if case["spread"]:
        counts = (uniform(W) * (case["per_worker"] + 1)).floor().to(torch.int64)
    else:
        counts = torch.full((W,), case["per_worker"], dtype=torch.int64, device="cuda")
    off = torch.zeros(W + 1, dtype=torch.int32, device="cuda")
    off[1:] = counts.cumsum(0)
    n = int(off[-1])
    d = dict(off=off, rin=_lengths(gen, n, IN_LAW), rpred=_lengths(gen, n, out_law))
    d["rgen"] = torch.minimum((uniform(n) * d["rpred"]).floor().to(torch.int32), d["rpred"] - 1)
    rate = 0.36 + 0.16 * uniform(n)  # the share of the budget a token that was used so far
    d["tdec"] = (d["rgen"] * rate * 2.0 * case["T_dec"] * case["theta"]).to(torch.float32) if case["history"] else None
    for suffix, m in (("", case["cands"]), ("2", case["then_score"])):
        d["cin" + suffix] = _lengths(gen, m, IN_LAW)
        d["cpred" + suffix] = _lengths(gen, m, out_law)
        d["cwait" + suffix] = (uniform(m) * 100.0).to(torch.float32)
    return d


def _arrivals(case, seed):
    """Poisson arrivals whose rate swings 4:1 over the trace, with the recipe's lengths (host arrays)."""
    rng = np.random.default_rng(seed)
    n, peak = case["requests"], case["rate"]
    mean, amp = 0.625 * peak, 0.375 * peak
    span = n / mean
    t = np.cumsum(rng.exponential(1.0 / peak, 4 * n + 4096))
    keep = rng.random(len(t)) * peak <= mean - amp * np.cos(2.0 * np.pi * t / span)
    t = t[keep][:n] * 1000.0

    def lengths(law):
        m, s, lo, hi = law
        return np.clip(np.rint(rng.lognormal(math.log(m) - 0.5 * s * s, s, n)), lo, hi).astype(np.int32)

    return t, lengths(IN_LAW), lengths(OUT_LAW)


def _place(x, memory):
    if x is None or memory == "device":
        return x
    return x.cpu().pin_memory() if memory == "pinned" else x.cpu().numpy()


def _empty(shape, dtype, memory):
    if memory == "device":
        return torch.zeros(shape, dtype=dtype, device="cuda")
    t = torch.zeros(shape, dtype=dtype)
    return t.pin_memory() if memory == "pinned" else t.numpy()


def prepare(case, seed):
    s = dict(case=case)
    if case["call"] in ("simulate", "search"):
        s["params"] = A.make_params(_params(case), case["slots"])
        s["trace"] = A.make_trace(*_arrivals(case, seed))
        gpus = [case["gpus"]] if case["call"] == "simulate" else list(GPU_MIX)
        s["cfgs"] = A.make_cfgs(gpus, [g * case["kv"] for g in gpus], [1.0 / math.sqrt(g) for g in gpus])
        s["out"] = np.zeros(A.SIMULATE_OUT)
        s["n"] = np.zeros(len(gpus), np.int32)
        return s
    d = _requests(case, seed)
    gpus, kv, scale = _sizes(case)
    W, C, mem = case["workers"], case["cands"], case["memory"]
    none = np.zeros(0, np.int32)
    cl = A.Cluster(_params(case), gpus, kv, scale, case["slots"], np.zeros(W + 1, np.int32), none, none, none)
    s["cluster"] = cl
    s["state"] = [_place(d[k], mem) for k in ("off", "rin", "rgen", "rpred", "tdec")]
    s["cands"] = [_place(d[k], mem) for k in ("cin", "cpred", "cwait")]
    if case["call"] == "score":
        cl.load(*s["state"])
    if case["call"] == "round":
        s["placement"] = _empty(C, torch.int32, mem)
        s["count"] = np.zeros(W, np.int32)
        s["next"] = [_place(d[k], mem) for k in ("cin2", "cpred2", "cwait2")]
        C = case["then_score"]
    s["flags"] = _empty((C, W), torch.uint8, mem) if "f" in case["outputs"] and C else None
    s["margin"] = _empty((C, W), torch.float32, mem) if "m" in case["outputs"] and C else None
    s["argbest"] = _empty(C, torch.int32, mem) if "a" in case["outputs"] and C else None
    return s


def run(s):
    case, call = s["case"], s["case"]["call"]
    if call == "simulate":
        A.aladdin_simulate(s["params"], s["cfgs"][0], case["workers"], s["trace"], 100.0, 0, 0, s["out"])
        return {"out": s["out"]}
    if call == "search":
        best, total = A.aladdin_min_workers(s["params"], s["cfgs"], s["trace"], 100.0, case["workers"], s["n"])
        if best >= 0:
            A.aladdin_simulate(s["params"], s["cfgs"][best], s["n"][best], s["trace"], 100.0, 0, 1, s["out"])
        return {"n_workers": s["n"], "best": best, "total_gpus": total, "out": s["out"]}
    cl = s["cluster"]
    out = {}
    if call == "heartbeat":
        A.aladdin_cluster_load_score(cl.handle, *s["state"], case["cands"], *s["cands"], s["flags"], s["margin"],
                                     s["argbest"])
    elif call == "score":
        A.aladdin_score(cl.handle, case["cands"], *s["cands"], s["flags"], s["margin"], s["argbest"])
    else:
        cl.load(*s["state"])
        A.aladdin_place_round(cl.handle, case["cands"], *s["cands"], s["placement"])
        out["placement"] = s["placement"]
        if case["then_score"]:
            A.aladdin_score(cl.handle, case["then_score"], *s["next"], s["flags"], s["margin"], s["argbest"])
        # the requests each worker now holds: what the dispatcher reports
        A.aladdin_cluster_state(cl.handle, s["count"], None, None, None, None)
        out["count"] = s["count"]
    for k in ("flags", "margin", "argbest"):
        if s[k] is not None:
            out[k] = s[k]
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without.

PAIR_FLOPS = 20  # a pair's bounds, their minimum and the comparisons


def work(case):
    if case["call"] in ("simulate", "search"):
        n, fleets = case["requests"], 1 if case["call"] == "simulate" else len(GPU_MIX)
        return {"bytes": 16 * n, "flops": PAIR_FLOPS * n * case["workers"] * fleets}
    W, C = case["workers"], case["cands"]
    held = W * case["per_worker"] * (0.5 if case["spread"] else 1.0)
    per = ("f" in case["outputs"]) + 4 * ("m" in case["outputs"])
    scored = case["then_score"] if case["call"] == "round" else C
    size = held * (16 if case["history"] else 12) + 4 * (W + 1) + 12 * C + per * scored * W
    size += 4 * scored if "a" in case["outputs"] else 0
    if case["call"] == "round":
        size += 12 * scored + 4 * C + 4 * W
    return {"bytes": size, "flops": PAIR_FLOPS * W * (C + (scored if case["call"] == "round" else 0)) / case["groups"]}


def tolerance(case):
    # placements, counts and simulated schedules are whole decisions of the same rule
    if case["call"] in ("simulate", "search", "round") and not case.get("then_score"):
        return "exact"
    # margins: 32-bit roundings of the bounds, measured at up to 1.9e-7 (2-norm) and 9.9e-7 (largest) of the
    # 64-bit values over the ranges below; a flag or a choice may turn where a bound ties
    return {"rel": 8e-7, "max": 4e-6, "differ": 1e-5}


# ---------------------------------------------------------------------------
# The margins in 64 bits: the scheduler's constraints from their definition, per worker over the sorted
# remaining lengths.

def exact(case, seed):
    if case["call"] not in ("heartbeat", "score") or "m" not in case["outputs"]:
        return None
    d, p = _requests(case, seed), _params(case)
    _, kv, scale = _sizes(case)
    W, C, f8, dev = case["workers"], case["cands"], torch.float64, "cuda"
    k1, c1 = (p["k1"], p["c1"]) if case["phase"] == "mixed" else (0.0, 0.0)
    k2, c2, c3, h, jj = p["k2"], p["c2"], p["c3"], p["h"], p["j"]
    budget = p["theta"] * p["T_dec"]
    ca, cr, cw = d["cin"].to(f8), d["cpred"].to(f8), d["cwait"].to(f8)
    margin = torch.empty((C, W), dtype=f8, device=dev)
    inf = float("inf")
    off = d["off"].long()
    B = max(1, int((off[1:] - off[:-1]).max()))
    step = max(1, min(W, (1 << 25) // max(C, B)))
    for w0 in range(0, W, step):
        w1 = min(W, w0 + step)
        o, cnt = off[w0:w1], (off[w0 + 1:w1 + 1] - off[w0:w1])
        S = torch.tensor(scale[w0:w1], device=dev).to(f8)[:, None]
        M = torch.tensor(kv[w0:w1], device=dev).to(f8)[:, None]
        col = torch.arange(B, device=dev)[None, :]
        live = col < cnt[:, None]
        at = torch.where(live, o[:, None] + col, torch.zeros_like(col))
        zero = torch.zeros((w1 - w0, B), dtype=f8, device=dev)

        def take(x):
            return torch.where(live, x[at].to(f8), zero) if x.numel() else zero

        gen, pred, rin = take(d["rgen"]), take(d["rpred"]), take(d["rin"])
        bank = budget * gen - take(d["tdec"]) if d["tdec"] is not None else zero
        r = torch.where(live, pred - gen, torch.full_like(zero, 1e9))
        r, by = r.sort(dim=1)
        a, bank, ok = (rin + gen).gather(1, by), bank.gather(1, by), live.gather(1, by)
        r0 = torch.where(ok, r, zero)

        def sums(x):  # prefix sums with the empty prefix first
            return torch.cat([torch.zeros((w1 - w0, 1), dtype=f8, device=dev), x.cumsum(1)], 1)

        n_all = cnt[:, None].to(f8)
        PR, PRA, PA = sums(r0), sums(r0 * a + r0 * (r0 + 1) / 2), sums(a)
        k = torch.arange(B + 1, device=dev)[None, :].to(f8)
        N, Asuf = (n_all - k).clamp(min=0), PA[:, -1:] - PA

        def decode_time(x, i):  # time of x iterations over the latency scale, row i <= x
            g = [t.gather(1, i) for t in (PR, PRA, N, Asuf)]
            return c2 * g[0] + k2 * g[1] + x * (c3 + c2 * g[2] + k2 * g[3]) + k2 * g[2] * x * (x + 1) / 2

        own = (torch.arange(B, device=dev)[None, :] + 1).expand(w1 - w0, B)
        sigma = budget * r0 + bank - S * decode_time(r0, own)
        u = sigma - S * (c2 * r0 + k2 * r0 * (r0 + 1) / 2)
        KV = h * (Asuf[:, :-1] + r0 * N[:, :-1]) + jj * N[:, :-1]
        big = torch.full((w1 - w0, 1), inf, dtype=f8, device=dev)

        def prefix_min(x):
            return torch.cat([big, torch.where(ok, x, torch.full_like(x, inf)).cummin(1)[0]], 1)

        def suffix_min(x):
            return torch.cat([torch.where(ok, x, torch.full_like(x, inf)).flip(1).cummin(1)[0].flip(1), big], 1)

        PM, SM = -prefix_min(-(KV + h * r0)), -suffix_min(-KV)
        pre = prefix_min((u - S * c1) / (S * (k2 * r0.clamp(min=1) + k1)))
        suf = suffix_min(sigma)
        Rc = cr[None, :].expand(w1 - w0, C).contiguous()
        i = torch.searchsorted(r.contiguous(), Rc, right=True)
        n1 = N.gather(1, i) + 1
        bound = torch.floor((M - jj * n1) / h) - Asuf.gather(1, i) - Rc * n1
        bound = torch.minimum(bound, torch.floor((M - jj - PM.gather(1, i)) / h))
        bound = torch.where(SM.gather(1, i) > M, torch.full_like(bound, -inf), bound)
        if case["phase"] == "mixed":
            bound = torch.minimum(bound, (p["T_pre"] - cw[None, :]) / (S * k1) - c1 / k1)
        X = c2 * Rc + k2 * Rc * (Rc + 1) / 2
        if case["mode"] == "approx":
            saved = torch.where(ok, p["theta"] * (p["T_dec"] * gen - (take(d["tdec"]) if d["tdec"] is not None else p["T_dec"] * p["theta"] * gen)).gather(1, by),
                                torch.full_like(zero, inf)).min(1, keepdim=True)[0]
            if case["phase"] == "mixed":
                bound = torch.minimum(bound, (saved - S * c1) / (S * k1))
            held = (rin + p["gamma"] * pred).sum(1, keepdim=True)
            limit = (p["T_dec"] / S - c3 - c2 * (n_all + 1)) / k2
            bound = torch.minimum(bound, p["theta"] * limit - held - p["gamma"] * Rc)
        else:
            bound = torch.minimum(bound, pre.gather(1, i))
            bound = torch.minimum(bound, (suf.gather(1, i) / S - c1 - X) / (k2 * Rc + k1))
            bound = torch.minimum(bound, (budget * Rc / S - X - decode_time(Rc, i)) / (k2 * Rc))
        margin[:, w0:w1] = (bound - ca[None, :]).t()
    return {"flags": None, "margin": margin, "argbest": None}
