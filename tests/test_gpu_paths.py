"""Dispatch edges of the scoring and table-building kernels: a call on one side
of an edge gives, byte for byte, what the call on the other side gives for the
same pairs. Scoring of both kinds is compared with the oracle elsewhere; here
the sizes are the ones where the kernels change."""
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


def score_device(A, cl, wl, n, off=0, flags=True, margin=True):
    """Rows of the first n candidates on device buffers that start `off`
    elements into their allocation."""
    import torch
    dev = torch.device("cuda")
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x[:n])).to(dev)
    W = wl.n_workers
    f = torch.zeros(n * W + off, dtype=torch.uint8, device=dev)[off:]
    m = torch.zeros(n * W + off, dtype=torch.float32, device=dev)[off:]
    a = torch.zeros(n, dtype=torch.int32, device=dev)
    A.aladdin_score(cl.handle, n, d(wl.cand_in), d(wl.cand_pred), d(wl.cand_wait),
                    f if flags else None, m if margin else None, a)
    torch.cuda.synchronize()
    return (f.cpu().numpy().reshape(n, W), m.cpu().numpy().reshape(n, W), a.cpu().numpy())


# pairs around 2^20 and workers around 2,048, whole and ragged rows of 16 and 4
@pytest.mark.parametrize("W,n,small,extra", [
    (1024, 1025, 1024, {}),
    (1023, 1100, 1025, {}),
    (2048, 513, 512, {}),
    (2046, 700, 512, dict(mode=1, theta=0.9)),
    (1001, 1300, 7, dict(phase=1)),
    (1, 2000, 1, {}),
    (2049, 600, 600, {}),
])
def test_scoring_paths_agree(A, synth, W, n, small, extra):
    """More pairs than the one-launch path takes (sorted, tiled) against fewer
    (direct), aligned and unaligned outputs, each output alone; with pending
    requests, refused candidates and every length of the candidates' law."""
    wl = synth.make_cluster("paths", 900 + W, W, 30, 40000, n, per_worker_random=True, b_cap=128,
                            params=dict(T_pre=150.0, T_dec=22.0, **extra))
    tdec = synth.decode_history(wl, 8.0, 20.0, 5)
    with A.Cluster.from_workload(wl, tdec_ms=tdec) as cl:
        cl.place_round(wl.cand_in[:60], wl.cand_pred[:60], wl.cand_wait[:60])
        wl.cand_pred[3::29] = 0
        full = score_device(A, cl, wl, n)
        valid = wl.cand_pred > 0
        assert np.array_equal(full[0] == A.FLAG_INVALID, np.broadcast_to(~valid[:, None], (n, W)))
        assert W == 1 or 0 < (full[0][valid] == A.FEASIBLE).mean() < 1
        few = score_device(A, cl, wl, small)
        for x, y in zip(few, full):
            assert x.tobytes() == y[:small].tobytes()
        for off in (1, 3):
            for x, y in zip(score_device(A, cl, wl, n, off), full):
                assert x.tobytes() == y.tobytes(), off
        for k in (n, small):
            f = score_device(A, cl, wl, k, flags=True, margin=False)
            m = score_device(A, cl, wl, k, flags=False, margin=True)
            assert f[0].tobytes() == full[0][:k].tobytes()
            assert m[1].tobytes() == full[1][:k].tobytes()
            assert f[2].tobytes() == m[2].tobytes() == full[2][:k].tobytes()


@pytest.mark.parametrize("cap", [32, 64, 128, 256, 512, 1024])
def test_table_builds_agree(A, synth, cap):
    """608 workers (one CTA of cooperating warps each) against 609 (a warp each,
    and a list of those beyond 128 requests), with workers at the edges of the
    warps' shares: the shared workers' pairs are the same bytes."""
    W, n = 609, 50
    per = min(cap, 200)
    wl = synth.make_cluster("builds", 950 + cap, W, per, 60000 + 700 * cap, n,
                            per_worker_random=True, b_cap=cap,
                            params=dict(T_pre=900.0, T_dec=20.0 + 0.15 * cap))
    counts = np.diff(wl.roff)
    for i, c in enumerate((0, 1, 31, 32, 33, 64, 127, 128, 129, 255, 256, 257, 511, 512, 1023)):
        if c <= cap:
            counts[i * 40] = c
    counts[607] = cap
    rng = np.random.default_rng(cap)
    roff = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    N = int(roff[-1])
    inp = rng.integers(16, 900, N).astype(np.int32)
    pred = rng.integers(8, 700, N).astype(np.int32)
    gen = rng.integers(0, pred).astype(np.int32)
    got = []
    for k in (W, W - 1):
        m = int(roff[k])
        with A.Cluster(wl.params, wl.gpus[:k], wl.kv_capacity[:k], wl.lat_scale[:k], cap,
                       roff[:k + 1], inp[:m], gen[:m], pred[:m]) as cl:
            assert cl.status() == A.OK
            got.append(cl.score(wl.cand_in, wl.cand_pred, wl.cand_wait, detail=True))
    for key in ("flags", "margin", "kvpeak", "tcand"):
        a, b = got[0][key], got[1][key]
        if a.ndim == 2 and a.shape[1] == W:
            a = a[:, :W - 1]
        assert np.ascontiguousarray(a).tobytes() == b.tobytes(), key
    assert 0 < (got[0]["flags"] == A.FEASIBLE).mean() < 1
