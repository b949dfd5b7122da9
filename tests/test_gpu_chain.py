"""The placement chain (k_round_chain) at the sizes where it changes shape:
tables of each size class whose workers cross the register steps, rounds with
and without the flag matrix, groups, every option that changes a bound, and
simulations; against the oracle, through the C ABI."""
import numpy as np
import pytest

from parity import compare_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_2405_06856_gb300 import build
    build.build()
    from paper_2405_06856_gb300 import aladdin
    return aladdin


LOOSE = dict(T_pre=1e5, T_dec=400.0)
REFUSED = -2
HIST = dict(lo_ms=8.0, hi_ms=20.0)

# W, slots, requests a worker at first (at most), KV, candidates, parameters.
# A hot worker's lanes hold one request more at every 128 (at every 256 on 1,024
# slots, where 129 to 511 requests are staged), so the first rows fill
# workers across those counts; the others are the dispatch's edges (64 workers,
# 4,096 pairs a call) and the options.
ROUNDS = {
    "slots32": (40, 32, 8, 9000, 300, dict(T_pre=200.0)),
    "slots128": (12, 128, 60, 50000, 500, LOOSE),
    "slots256-over-128": (6, 256, 120, 105000, 500, LOOSE),
    "slots512-over-128-256-384": (4, 512, 250, 240000, 900, LOOSE),
    "slots1024-over-256-384-512": (3, 1024, 380, 420000, 1500, LOOSE),
    "slots1024-fill": (8, 1024, 10, 60000, 900, dict(T_pre=150.0)),
    "table-63-workers": (63, 128, 30, 40000, 200, dict(T_pre=300.0, T_dec=20.0)),
    "flags-64-workers": (64, 128, 30, 40000, 200, dict(T_pre=300.0, T_dec=20.0)),
    "table-4095-pairs": (195, 128, 30, 40000, 31, dict(T_pre=300.0, T_dec=20.0)),
    "flags-4096-pairs": (256, 128, 30, 40000, 24, dict(T_pre=300.0, T_dec=20.0)),
    "flags-many-words": (1100, 64, 20, 20000, 600, dict(T_pre=200.0, T_dec=11.0)),
    "one-candidate": (20, 128, 30, 40000, 1, {}),
    "one-worker-fills": (1, 256, 30, 30000, 150, LOOSE),
    "groups3": (100, 256, 40, 60000, 400, dict(groups=3, T_dec=30.0)),
    "groups7-ragged-fill": (17, 512, 40, 30000, 600, dict(groups=7, T_dec=30.0)),
    "gamma-h-j": (60, 256, 40, 90000, 300, dict(gamma=0.3, h=2, j=3, T_pre=400.0, T_dec=24.0)),
    "theta-history": (60, 256, 40, 90000, 300, dict(theta=0.85, T_pre=400.0, T_dec=26.0, hist=1)),
    "approx-history": (60, 256, 40, 90000, 300,
                       dict(mode=1, theta=0.9, T_pre=200.0, T_dec=26.0, hist=1)),
    "approx-flags": (260, 256, 40, 90000, 300,
                     dict(mode=1, theta=0.9, T_pre=200.0, T_dec=26.0, hist=1)),
    "decode": (60, 256, 40, 90000, 300, dict(phase=1, T_dec=26.0, hist=1)),
    "flags-misses": (2600, 32, 20, 9000, 400, dict(T_pre=200.0)),
    "table-misses": (63, 32, 20, 9000, 64, dict(T_pre=200.0)),
    "flags-fresh-start": (1200, 32, 20, 9000, 2250, dict(T_pre=200.0)),  # over 256 workers modified
}


def workload(synth, name):
    W, cap, per, kv, n, p = ROUNDS[name]
    p = dict(p)
    hist = p.pop("hist", 0)
    seed = 700 + list(ROUNDS).index(name)
    wl = synth.make_cluster("chain", seed, W, per, kv, n, per_worker_random=True, b_cap=cap,
                            gpus_cycle=(1, 2) if "history" in name else (1,), params=p)
    wl.cand_pred[max(n // 2, 1)::17] = 0  # refused candidates inside the runs
    return wl, synth.decode_history(wl, HIST["lo_ms"], HIST["hi_ms"], seed) if hist else None


def oracle_cluster(orc, wl, tdec):
    return orc.Cluster.from_workload(wl, tdec=None if tdec is None else tdec.astype(np.float64))


def oracle_round(oc, wl, lo, hi):
    """Candidates [lo, hi); the refused ones are not handed to the oracle."""
    c = np.arange(lo, hi)
    ok = wl.cand_pred[lo:hi] > 0
    out = np.full(hi - lo, REFUSED, np.int32)
    out[ok] = oc.place_round(wl.cand_in[c[ok]], wl.cand_pred[c[ok]], wl.cand_wait[c[ok]], crid=c[ok])
    return out


@pytest.mark.parametrize("name", list(ROUNDS))
def test_chain_places_like_the_oracle(A, orc, synth, name):
    """Two calls of one open round, and scoring against the tables that the
    chain left (no pair that decides a placement here is within the fp32 bar of
    zero)."""
    wl, tdec = workload(synth, name)
    n = wl.n_cand
    oc = oracle_cluster(orc, wl, tdec)
    cut = n - n // 3
    if name.endswith("-pairs"):  # the first call's pairs, at the edge of the dispatch
        assert wl.n_workers * cut == int(name.split("-")[1])
    with A.Cluster.from_workload(wl, tdec_ms=tdec) as cl:
        pl, rl = [], []
        for lo, hi in ((0, cut), (cut, n)):
            if lo == hi:
                continue
            q = (wl.cand_in[lo:hi], wl.cand_pred[lo:hi], wl.cand_wait[lo:hi])
            pl.append(cl.place_round(*q))
            rl.append(oracle_round(oc, wl, lo, hi))
        assert cl.status() == A.OK
        pl, rl = np.concatenate(pl), np.concatenate(rl)
        mis = np.flatnonzero(pl != rl)
        assert len(mis) == 0, (mis[0], pl[mis[0]], rl[mis[0]])
        assert (pl >= 0).any()
        k = min(n, 40)
        ok = wl.cand_pred[:k] > 0
        q = (wl.cand_in[:k][ok], wl.cand_pred[:k][ok], wl.cand_wait[:k][ok])
        g = cl.score(*q, detail=True)
        compare_pairs(oc.score(*q), g["flags"], g["margin"], q[0], g["kvpeak"], g["tcand"], name)
        counts = cl.state()[0]
        assert np.array_equal(counts, oc.n)


def kv_peak(wl, w):
    """KV usage of worker w's requests at its highest."""
    q = slice(wl.roff[w], wl.roff[w + 1])
    r = np.sort(wl.req_pred[q] - wl.req_gen[q])
    a = (wl.req_in[q] + wl.req_gen[q])[np.argsort(wl.req_pred[q] - wl.req_gen[q])]
    left = np.arange(len(r), 0, -1)
    return int((np.cumsum(a[::-1])[::-1] + r * left).max())


def test_chain_counts_at_the_staging_lines(A, orc, synth):
    """On 1,024 slots who loads a worker that becomes hot depends on how many
    requests it holds: the look-ahead warps from 129 to 511, its own warps
    otherwise. Every worker of a direct round becomes hot with a count at
    those lines, and some again after they left."""
    counts = np.array([126, 127, 128, 129, 130, 510, 511, 512, 513, 128, 511, 0], np.int64)
    W, n = len(counts), 120
    wl = synth.make_cluster("lines", 811, W, 520, 1, n, b_cap=1024, params=LOOSE)
    rows = np.concatenate([np.arange(wl.roff[w], wl.roff[w] + counts[w]) for w in range(W)])
    for k in ("req_in", "req_gen", "req_pred"):
        setattr(wl, k, getattr(wl, k)[rows].copy())
    wl.roff = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    wl.kv_capacity = np.array([(kv_peak(wl, w) if counts[w] else 0) + 2500 for w in range(W)], np.int64)
    oc = oracle_cluster(orc, wl, None)
    ref = oracle_round(oc, wl, 0, n)
    assert set(ref[ref >= 0]) == set(range(W))  # every count becomes hot
    with A.Cluster.from_workload(wl) as cl:
        pl = cl.place_round(wl.cand_in, wl.cand_pred, wl.cand_wait)
        assert cl.status() == A.OK
        assert np.array_equal(pl, ref), np.argwhere(pl != ref)[:5]
        assert np.array_equal(cl.state()[0], oc.n)


@pytest.mark.parametrize("W", [512, 513, 2560, 2561, 4608, 4609, 5120])
def test_chain_finds_the_last_workers(A, orc, synth, W):
    """Every worker but the lightest is full: the scan of a candidate's flags
    runs to the end of the row, at the edges of its steps."""
    n = 40
    wl = synth.make_cluster("last", W, W, 3, 1, n, b_cap=32, params=LOOSE)
    empty = np.array([0, W // 2, W - 1])
    keep = np.repeat(~np.isin(np.arange(W), empty), 3)
    for k in ("req_in", "req_gen", "req_pred"):
        setattr(wl, k, getattr(wl, k)[keep].copy())
    wl.roff = np.concatenate([[0], np.cumsum(np.where(np.isin(np.arange(W), empty), 0, 3))]).astype(np.int32)
    wl.kv_capacity = np.where(np.isin(np.arange(W), empty), 6000, 10).astype(np.int64)
    oc = oracle_cluster(orc, wl, None)
    ref = oracle_round(oc, wl, 0, n)
    assert set(ref) == {-1, *empty}
    with A.Cluster.from_workload(wl) as cl:
        pl = cl.place_round(wl.cand_in, wl.cand_pred, wl.cand_wait)
        assert np.array_equal(pl, ref), np.argwhere(pl != ref)[:5]


@pytest.mark.parametrize("cap", [128, 512, 1024])
@pytest.mark.parametrize("extra", [{}, dict(mode=1, theta=0.9), dict(gamma=0.3, h=2, j=3, k1=0.0011, k2=1.7e-4,
                                                                    c2=0.047, c3=7.3)])
def test_chain_tables_equal_built_ones(A, synth, cap, extra):
    """The chain forms the tables of the workers it used from its own sums; a
    restored cluster builds them from the requests. On workers of several
    latency scales both score, place and execute alike, byte for byte."""
    p = dict(dict(T_pre=300.0, T_dec=12.0), **extra)
    wl = synth.make_cluster("built", 900 + cap, 96, 20, 60000, 1600, per_worker_random=True, b_cap=cap,
                            gpus_cycle=(1, 2, 4) if cap == 128 else (1, 2, 4, 8), params=p)
    h = synth.decode_history(wl, 8.0, 12.0, 5)
    with A.Cluster.from_workload(wl, tdec_ms=h) as a, A.Cluster.from_workload(wl, tdec_ms=h) as b:
        pl = a.place_round(wl.cand_in[:900], wl.cand_pred[:900], wl.cand_wait[:900])
        used = np.unique(pl[pl >= 0])
        assert len(used) > 8 and len(np.unique(wl.lat_scale[used])) >= 3
        A.aladdin_cluster_restore(b.handle, A.aladdin_cluster_save(a.handle))
        q = (wl.cand_in[900:1200], wl.cand_pred[900:1200], wl.cand_wait[900:1200])
        sa, sb = a.score(*q), b.score(*q)
        diff = np.argwhere(sa["margin"].view(np.int32) != sb["margin"].view(np.int32))
        assert len(diff) == 0, (len(diff), sa["margin"][tuple(diff[0])], sb["margin"][tuple(diff[0])])
        assert np.array_equal(sa["flags"], sb["flags"]) and np.array_equal(sa["argbest"], sb["argbest"])
        outs = []
        for cl in (a, b):
            pl = cl.place_round(wl.cand_in[900:], wl.cand_pred[900:], wl.cand_wait[900:])
            cl.advance(100.0)
            outs.append([pl.tobytes()] + [x.tobytes() for x in cl.state()])
        assert outs[0] == outs[1]


@pytest.mark.parametrize("N,cap,kv,rate,extra", [
    (7, 64, 16000, 30.0, {}),
    (6, 128, 40000, 60.0, dict(gamma=0.3)),
    (5, 512, 120000, 120.0, dict(T_dec=40.0)),
    (3, 1024, 300000, 160.0, dict(T_dec=80.0)),
    (9, 256, 40000, 60.0, dict(rebalance=1, theta=0.9)),
    (2047, 32, 6000, 3000.0, dict(T_dec=14.0)),
    (2049, 32, 6000, 3000.0, dict(T_dec=14.0)),
    # both sides of the lines past which the sliced round serves
    (192, 128, 6000, 3000.0, dict(T_dec=14.0)),
    (193, 128, 6000, 3000.0, dict(T_dec=14.0)),
    (224, 256, 6000, 3000.0, dict(T_dec=14.0)),
    (225, 256, 6000, 3000.0, dict(T_dec=14.0)),
    (448, 512, 3000, 4000.0, dict(T_dec=14.0)),
    (449, 512, 3000, 4000.0, dict(T_dec=14.0)),
    (384, 1024, 3000, 4000.0, dict(T_dec=14.0)),
    (385, 1024, 3000, 4000.0, dict(T_dec=14.0)),
])
def test_chain_simulates_like_the_oracle(A, orc, synth, N, cap, kv, rate, extra):
    tr = synth.diurnal_trace(40 + N, 700, rate, rate / 4)
    p = dict(synth.BASE_PARAMS, **extra)
    ref = orc.simulate(p, N, cap, kv, 1.0, tr, 100.0, stop_at_fail=False, drain=True)
    out = np.zeros(A.SIMULATE_OUT)
    A.aladdin_simulate(A.make_params(p, cap), A.make_cfgs([1], [kv], [1.0])[0], N,
                       A.trace_of(tr), 100.0, 0, 1, out)
    assert int(out[0]) == ref["failed"] and int(out[1]) == ref["placed"], (out, ref)
    assert int(out[2]) == ref["heartbeats"] and int(out[5]) == ref["violations"], (out, ref)
    assert out[3] == pytest.approx(ref["max_ttft"], rel=1e-12)
    assert out[4] == pytest.approx(ref["max_atgt"], rel=1e-12)
    assert int(out[8]) == ref["moved"]


def test_exact_predictions_equal_real_lengths(A, synth):
    """The execution step has a branch of its own where predictions are exact;
    a trace that states the same lengths as the real ones takes the general
    branch and must end with the same numbers, bit for bit."""
    tr = synth.diurnal_trace(77, 1500, 80.0, 20.0)
    p = dict(synth.BASE_PARAMS, T_dec=30.0)
    outs = []
    for real in (None, np.asarray(tr.req_pred)):
        t = synth.Trace(tr.t_arr, tr.req_in, tr.req_pred, real, None)
        out = np.zeros(A.SIMULATE_OUT)
        A.aladdin_simulate(A.make_params(p, 256), A.make_cfgs([1], [40000], [1.0])[0], 6,
                           A.trace_of(t), 100.0, 0, 1, out)
        outs.append(out)
    assert outs[0][1] > 0 and outs[0].tobytes() == outs[1].tobytes()
