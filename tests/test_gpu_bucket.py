"""The bucket-major scan of large batches (kernels_bucket.cu) against the
per-query scan (explicit CTA layout) and the oracle: ids and distance bits are
equal. eps0 = 0 makes every bound the estimate itself, so that one wrong
product changes which codes survive."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2405_12497_gb300 import rabitq
    return rabitq


def _mix(rng, n, d, comps=40):
    mu = rng.standard_normal((comps, d))
    return (mu[rng.integers(0, comps, n)] + 0.6 * rng.standard_normal((n, d))).astype(np.float32)


def _same(R, G, Q, k, nprobe, **kw):
    import torch
    qd = torch.from_numpy(Q).cuda()
    ids, dist = G.search(qd, k, nprobe, **kw)
    ref_i, ref_d = G.search(qd, k, nprobe, layout=R.LAYOUT_CTA, staging=R.STAGING_OFF, **kw)
    assert torch.equal(ids, ref_i)
    assert torch.equal(dist.view(torch.int32), ref_d.view(torch.int32))
    return ids.cpu().numpy(), dist.cpu().numpy()


# code lengths: one operand stage, a half stage, several, the 16-pair items of
# the longest; d below the code length (padding)
@pytest.mark.parametrize("d,bits", [(50, 64), (128, 128), (100, 192), (256, 256), (300, 320),
                                    (420, 448), (960, 1024), (2000, 2048), (4000, 4096)])
def test_code_lengths(R, d, bits):
    rng = np.random.default_rng(bits)
    n = 9000 if d <= 512 else 3000
    data, Q = _mix(rng, n, d), _mix(rng, 1000, d)
    G = R.Index.build(data, 24, seed=2, code_bits=bits, kmeans_iters=3)
    for k, nprobe, eps0 in ((10, 5, 0.0), (100, 7, 1.9), (1, 24, 0.5)):
        _same(R, G, Q, k, nprobe, eps0=eps0)


@pytest.mark.parametrize("metric", ["l2", "ip", "cosine"])
@pytest.mark.parametrize("bq", [1, 3, 4])
def test_metrics_and_bits(R, metric, bq):
    rng = np.random.default_rng(7)
    data, Q = _mix(rng, 8000, 128), _mix(rng, 1003, 128)
    G = R.Index.build(data, 32, seed=2, kmeans_iters=3, metric=metric)
    for k, nprobe in ((1, 3), (20, 9), (256, 32)):
        _same(R, G, Q, k, nprobe, bq=bq)
        _same(R, G, Q, k, nprobe, bq=bq, eps0=0.0)


# batch and bucket edges: 1000 is the smallest batch; K = 1 is one bucket of
# many tiles and several items, K = 1000 buckets of three codes with a few
# pairs each (fewer than k codes probed: pads), 1031 odd
@pytest.mark.parametrize("nq,K,nprobe,k", [(1000, 16, 4, 10), (1031, 1, 1, 100),
                                           (1031, 1000, 16, 64), (1000, 3, 3, 256),
                                           (2000, 700, 2, 10)])
def test_batch_edges_match_the_oracle(R, oracle_mod, nq, K, nprobe, k):
    from paper_2405_12497_gb300 import synth
    data, Q = synth.tiny(n=3000, nq=nq)
    G = R.Index.build(data, K, seed=2, kmeans_iters=3)
    ids, dist = _same(R, G, Q, k, nprobe)
    O = oracle_mod.OracleIndex(data, K=K, seed=2, iters=3)
    m = min(nq, 120)
    ids_o, dist_o = O.search(Q[:m], k, nprobe)
    assert np.array_equal(ids[:m], ids_o)
    assert np.array_equal(dist[:m].view(np.uint32), dist_o.view(np.uint32))


def test_ties_counts_and_plans(R):
    """Identical points (every bound equal), per-query probe counts, and a
    plan's replay, once below the batch rule."""
    import torch
    rng = np.random.default_rng(3)
    data = np.repeat(_mix(rng, 40, 128), 150, axis=0)
    Q = _mix(rng, 1100, 128)
    G = R.Index.build(data, 20, seed=2, kmeans_iters=3)
    _same(R, G, Q, 100, 6)
    npq = torch.from_numpy(rng.integers(1, 12, 1100).astype(np.int32)).cuda()
    _same(R, G, Q, 30, 11, per_query_nprobe=npq)
    plan = R.Plan(G, 100, 6, 1100)
    ids, dist = G.search(Q, 100, 6, layout=R.LAYOUT_CTA)
    for nq in (1100, 90, 1000):
        i, x = plan.search(Q[:nq])
        assert np.array_equal(i, ids[:nq]) and np.array_equal(x.view(np.uint32),
                                                              dist[:nq].view(np.uint32))


def test_long_lists_are_redone(R):
    """A bound so wide that every code of 16k-code buckets is a candidate: the
    lists (8192 entries for k <= 32) overflow and the per-query scan takes
    those queries."""
    rng = np.random.default_rng(5)
    data, Q = _mix(rng, 33000, 64, comps=2), _mix(rng, 1000, 64, comps=2)
    G = R.Index.build(data, 2, seed=2, kmeans_iters=2)
    _same(R, G, Q, 10, 1, eps0=40.0)


# a query whose squared norm overflows (every distance infinite: the lowest
# ids), one near the limit and one with a NaN, among ordinary ones; probe lists
# by a warp per query and, above 64 probes, by a CTA
@pytest.mark.parametrize("nprobe", [9, 70])
def test_overflowing_queries_leave_the_batch_alone(R, oracle_mod, nprobe):
    from paper_2405_12497_gb300 import synth
    data, Q = synth.tiny(n=6000, nq=1100)
    Q = Q.copy()
    unit = Q / np.linalg.norm(Q, axis=1, keepdims=True)
    Q[7], Q[300], Q[1099] = unit[7] * 1e20, unit[300] * 4e18, unit[1099] * 3e17
    G = R.Index.build(data, 100, seed=2, kmeans_iters=3)
    ids, dist = _same(R, G, Q, 10, nprobe)
    O = oracle_mod.OracleIndex(data, K=100, seed=2, iters=3)
    rows = [*range(60), 300, *range(1050, 1100)]
    for i in rows:  # (the quantization stream is the query's index in the call)
        t = O.trace(Q[i], i, 10, nprobe)
        assert np.array_equal(ids[i], t["ids"]), i
        assert np.array_equal(dist[i].view(np.uint32), t["dist"].view(np.uint32)), i
    bad = Q.copy()
    bad[500, 3] = np.nan
    with pytest.raises(Exception, match="non-finite"):
        G.search(bad, 10, nprobe)
    plan = R.Plan(G, 10, nprobe, 1100)
    pi, pd = plan.search(bad)
    ok = np.arange(1100) != 500
    assert np.array_equal(pi[ok], ids[ok])
    assert np.array_equal(pd[ok].view(np.uint32), dist[ok].view(np.uint32))


def test_few_long_lists_do_not_hold_up_a_batch(R):
    """Most queries probe two buckets, eight probe all 128 and have candidate
    lists of several times the even share: there is room for them, so they are
    not redone one by one (1.2 times the per-query scan's time when they are,
    0.4 times when not)."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    data = torch.randn((200_000, 64), generator=g, device="cuda")
    Q = torch.randn((1500, 64), generator=g, device="cuda")
    G = R.Index.build(data, 128, seed=2, kmeans_iters=3)
    npq = torch.full((1500,), 2, dtype=torch.int32, device="cuda")
    npq[::187] = 128

    def best(**kw):
        times = []
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            out = G.search(Q, 10, 128, per_query_nprobe=npq, max_candidates=1 << 19, **kw)
            e1.record()
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        return min(times[1:]), out

    t, (ids, dist) = best()
    t_ref, (ids_r, dist_r) = best(layout=R.LAYOUT_CTA, staging=R.STAGING_OFF)
    assert torch.equal(ids, ids_r)
    assert torch.equal(dist.view(torch.int32), dist_r.view(torch.int32))
    assert t < 0.9 * t_ref


# batches whose scan is too short to pay for the bucket-major launches: AUTO is
# no slower than the per-query scan (1.3 to 1.6 times its time where it took the
# other one)
@pytest.mark.parametrize("metric,K,k,nprobe", [("l2", 256, 100, 4), ("l2", 256, 256, 8),
                                               ("ip", 1024, 100, 16)])
def test_short_scans_stay_per_query(R, metric, K, k, nprobe):
    import torch
    rng = np.random.default_rng(4)
    data, Q = _mix(rng, 100_000, 96, comps=1000), _mix(rng, 1000, 96, comps=1000)
    G = R.Index.build(data, K, seed=2, code_bits=128, kmeans_iters=3, metric=metric)

    def best(**kw):
        plan = R.Plan(G, k, nprobe, 1000, **kw)
        plan.queries.copy_(torch.from_numpy(Q).cuda())
        times = []
        for _ in range(12):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            plan.run(1000)
            e1.record()
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        plan.sync()
        return min(times[2:])

    t, t_ref = best(), best(layout=R.LAYOUT_CTA, staging=R.STAGING_OFF)
    assert t < 1.1 * t_ref
