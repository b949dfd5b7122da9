"""Parity of distributed grouped scheduling (Appendix A) with the oracle,
through the C ABI: placements stay in their group, simulations and worker
searches with G groups match, Algorithm 2 moves within the group."""
import numpy as np
import pytest

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


def fresh_oracle(orc, wl):
    oc = orc.Cluster.from_workload(wl)
    oc.tdec[:] = wl.params["theta"] * wl.params["T_dec"] * oc.gen
    oc.has_tdec = True
    return oc


@pytest.mark.parametrize("policy", [0, 1, 2])
def test_grouped_rounds_match_oracle(A, orc, synth, policy):
    """Two rounds (request ids continue across calls) on 3 groups. With these
    round-decimal coefficients some slacks are exactly zero in fp64; where
    fp32 decides such a pair the other way the placements may diverge, and
    the first divergence must be such a near pair of the candidate's group
    (best-fit; JSQ and power of two test no feasibility and match exactly)."""
    wl = synth.config("w256", n_cand=1200, b_cap=128,
                      params=dict(T_dec=24.0, policy=policy, groups=3, seed=5))
    oc = fresh_oracle(orc, wl)
    with A.Cluster.from_workload(wl) as cl:
        pa = cl.place_round(wl.cand_in[:500], wl.cand_pred[:500], wl.cand_wait[:500])
        pb = cl.place_round(wl.cand_in[500:], wl.cand_pred[500:], wl.cand_wait[500:])
    ra = oc.place_round(wl.cand_in[:500], wl.cand_pred[:500], wl.cand_wait[:500],
                        crid=np.arange(500))
    rb = oc.place_round(wl.cand_in[500:], wl.cand_pred[500:], wl.cand_wait[500:],
                        crid=np.arange(500, 1200))
    pl, rl = np.concatenate([pa, pb]), np.concatenate([ra, rb])
    ok = pl >= 0
    assert ok.mean() > 0.2
    assert np.all(pl[ok] % 3 == np.arange(1200)[ok] % 3)
    mis = np.flatnonzero(pl != rl)
    if policy != 0:
        assert len(mis) == 0
    elif len(mis):
        c = int(mis[0])
        assert c > 100                       # a long exact prefix
        o2 = fresh_oracle(orc, wl)
        o2.place_round(wl.cand_in[:c], wl.cand_pred[:c], wl.cand_wait[:c], crid=np.arange(c))
        r = o2.score(wl.cand_in[c:c + 1], wl.cand_pred[c:c + 1], wl.cand_wait[c:c + 1])
        ws = np.arange(256)[np.arange(256) % 3 == c % 3]
        assert (r["near"][0, ws] <= 1e-5).any()


@pytest.mark.parametrize("policy,G", [(0, 2), (0, 5), (1, 3), (2, 4)])
def test_grouped_simulation_matches_oracle(A, orc, synth, policy, G):
    tr = synth.diurnal_trace(13, 1500, 60.0, 15.0)
    p = dict(synth.BASE_PARAMS, T_dec=30.0, policy=policy, groups=G, seed=8)
    for N in (5, 9):
        ref = orc.simulate(p, N, 256, 40000, 1.0, tr, 100.0, stop_at_fail=False, drain=True)
        out = np.zeros(A.SIMULATE_OUT)
        A.aladdin_simulate(A.make_params(p, 256), A.make_cfgs([1], [40000], [1.0])[0], N,
                           A.trace_of(tr), 100.0, 0, 1, out)
        lab = (policy, G, N, out, ref)
        assert int(out[0]) == ref["failed"] and int(out[1]) == ref["placed"], lab
        assert int(out[2]) == ref["heartbeats"] and int(out[5]) == ref["violations"], lab
        assert out[3] == pytest.approx(ref["max_ttft"], rel=1e-12), lab
        assert out[4] == pytest.approx(ref["max_atgt"], rel=1e-12), lab


def test_grouped_search_and_rebalance(A, orc, synth):
    tr = synth.diurnal_trace(6, 600, 60.0, 15.0)
    for G in (1, 3):
        p = dict(synth.BASE_PARAMS, T_dec=30.0, groups=G)
        ref = orc.min_workers(p, [1], [32768], [1.0], 256, tr, 100.0, 64)
        got = np.zeros(1, np.int32)
        A.aladdin_min_workers(A.make_params(p, 256), A.make_cfgs([1], [32768], [1.0]),
                              A.trace_of(tr), 100.0, 64, got)
        assert np.array_equal(got, ref) and got[0] > 0
    te = synth.with_prediction_error(synth.diurnal_trace(9, 1500, 60.0, 15.0), 0.5, 9)
    p = dict(synth.BASE_PARAMS, T_dec=30.0, groups=2, rebalance=1)
    ref = orc.simulate(p, 6, 256, 40000, 1.0, te, 100.0, stop_at_fail=False, drain=True)
    out = np.zeros(A.SIMULATE_OUT)
    A.aladdin_simulate(A.make_params(p, 256), A.make_cfgs([1], [40000], [1.0])[0], 6,
                       A.trace_of(te), 100.0, 0, 1, out)
    assert int(out[0]) == ref["failed"] and int(out[8]) == ref["moved"] and ref["moved"] > 0


def test_grouped_round_full_worker_stops_its_group(A, orc, synth):
    """Two groups of one worker (32 slots): group 0's worker holds 31
    requests, so its second candidate finds it full and group 0 stops; group 1
    places all of its candidates. The call reports ALADDIN_ERR_CAPACITY."""
    p = dict(synth.BASE_PARAMS, groups=2)
    roff = np.array([0, 31, 31], np.int32)
    args = (np.full(31, 100, np.int32), np.zeros(31, np.int32), np.full(31, 50, np.int32))
    cin, cpr = np.full(40, 100, np.int32), np.full(40, 50, np.int32)
    with A.Cluster(p, [1, 1], [10**6] * 2, [1.0] * 2, 32, roff, *args) as cl:
        pl = np.zeros(40, np.int32)
        with pytest.raises(A.AladdinError) as e:
            A.aladdin_place_round(cl.handle, 40, cin, cpr, None, pl)
        assert e.value.code == A.ERR_CAPACITY
        n = cl.state()[0]
    oc = orc.Cluster(p, [10**6] * 2, [1.0] * 2, 32, roff, *args)
    ref, full = oc.place_round(cin, cpr, crid=np.arange(40), allow_capacity=True)
    assert full and np.array_equal(pl, ref)
    assert list(pl[:4]) == [0, 1, -1, 1] and (pl[1::2] == 1).all() and (pl[2::2] == -1).all()
    assert list(n) == [32, 20] == list(oc.n)


@pytest.mark.parametrize("extra", [
    dict(phase=1, mode=1, groups=2, rebalance=1, theta=0.9),     # decode, approximate, Alg. 2
    dict(phase=1, policy=2, groups=3, seed=4),                  # decode, power of two
    dict(phase=0, mode=1, groups=3, rebalance=1, theta=0.85),   # mixed, approximate, Alg. 2
])
def test_features_compose(A, orc, synth, extra):
    """Decode instances, the approximate constraints, grouped scheduling,
    Algorithm 2 and prediction errors together: the simulation matches the
    oracle output for output."""
    te = synth.with_prediction_error(synth.diurnal_trace(21, 1200, 60.0, 15.0), 0.4, 21)
    p = dict(synth.BASE_PARAMS, T_dec=30.0, **extra)
    for N in (5, 8):
        ref = orc.simulate(p, N, 256, 40000, 1.0, te, 100.0, stop_at_fail=False, drain=True)
        out = np.zeros(A.SIMULATE_OUT)
        A.aladdin_simulate(A.make_params(p, 256), A.make_cfgs([1], [40000], [1.0])[0], N,
                           A.trace_of(te), 100.0, 0, 1, out)
        lab = (extra, N, out, ref)
        assert int(out[0]) == ref["failed"] and int(out[1]) == ref["placed"], lab
        assert int(out[2]) == ref["heartbeats"] and int(out[5]) == ref["violations"], lab
        assert out[3] == pytest.approx(ref["max_ttft"], rel=1e-12), lab
        assert out[4] == pytest.approx(ref["max_atgt"], rel=1e-12), lab
        assert int(out[6]) == ref["repredictions"] and int(out[7]) == ref["early_finishes"], lab
        assert int(out[8]) == ref["moved"], lab


@pytest.mark.parametrize("W,b_cap", [(8192, 32), (8194, 32), (6800, 1024), (8192, 1024)])
def test_grouped_rounds_of_large_groups(A, orc, synth, W, b_cap):
    """Two groups of 4,096 workers, the most that a placement chain holds (3,400
    on 1,024 slots are held without samples or limits), and of more, which
    k_round_grp places: like the oracle, over two calls."""
    wl = synth.make_cluster("large", W, W, 12, 9000, 90, per_worker_random=True, b_cap=b_cap,
                            params=dict(T_pre=200.0, T_dec=14.0, groups=2))
    oc = fresh_oracle(orc, wl)
    with A.Cluster.from_workload(wl) as cl:
        for lo, hi in ((0, 61), (61, 90)):
            q = wl.cand_in[lo:hi], wl.cand_pred[lo:hi], wl.cand_wait[lo:hi]
            pl = cl.place_round(*q)
            ref = oc.place_round(*q, crid=np.arange(lo, hi))
            assert np.array_equal(pl, ref), np.argwhere(pl != ref)[:5]
        assert (pl >= 0).any()
        assert np.array_equal(cl.state()[0], oc.n)


@pytest.mark.parametrize("b_cap,per,kv", [(32, 18, 6500), (128, 60, 22000), (1024, 60, 22000)])
@pytest.mark.parametrize("pg,G,n", [(1000, 3, 330), (700, 5, 505), (420, 2, 260)])
def test_groups_that_change_kernels(A, orc, synth, b_cap, per, kv, pg, G, n):
    """Nearly full groups past the line up to which the chain leads: the chains
    may leave the rest of a round to k_round_grp (which candidate it happens at
    depends on time); placements, state and scores are the oracle's. Only the KV
    limit binds, in integers, so that no pair is near."""
    wl = synth.make_cluster("change", 60 + b_cap + pg, pg * G, per, kv, n, per_worker_random=True,
                            b_cap=b_cap, params=dict(T_pre=1e5, T_dec=400.0, groups=G))
    oc = fresh_oracle(orc, wl)
    with A.Cluster.from_workload(wl) as cl:
        cut = n - n // 5
        for lo, hi in ((0, cut), (cut, n)):
            q = wl.cand_in[lo:hi], wl.cand_pred[lo:hi], wl.cand_wait[lo:hi]
            pl = cl.place_round(*q)
            ref = oc.place_round(*q, crid=np.arange(lo, hi))
            assert np.array_equal(pl, ref), np.argwhere(pl != ref)[:5]
        assert np.array_equal(cl.state()[0], oc.n)
        q = wl.cand_in[:20], wl.cand_pred[:20], wl.cand_wait[:20]
        s, r = cl.score(*q), oc.score(*q)
        assert np.array_equal(s["flags"] & 1, r["flags"] & 1)


def test_large_group_full_worker_stops_its_group(A, synth):
    """A full worker among 4,097 of its group: the error, the candidates placed
    before it, -1 from it on, and the other group's round to its end."""
    W, n = 8194, 9
    wl = synth.make_cluster("full", 3, W, 1, 10**6, n, b_cap=32,
                            params=dict(T_pre=1e6, T_dec=1e6, groups=2))
    counts = np.zeros(W, np.int64)
    counts[[4, 5]] = 30, 3
    rows = np.concatenate([np.arange(30), 30 + np.arange(3)])
    for k in ("req_in", "req_gen", "req_pred"):
        setattr(wl, k, getattr(wl, k)[rows].copy())
    wl.roff = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    pl = np.full(n, 7, np.int32)
    with A.Cluster.from_workload(wl) as cl:
        with pytest.raises(A.AladdinError) as e:
            A.aladdin_place_round(cl.handle, n, wl.cand_in, wl.cand_pred, wl.cand_wait, pl)
        assert e.value.code == A.ERR_CAPACITY
        assert pl.tolist() == [4, 5, 4, 5, -1, 5, -1, 5, -1]
        assert cl.state()[0][[4, 5]].tolist() == [32, 7]
