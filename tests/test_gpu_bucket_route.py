"""Which batches the bucket-major scan takes, as plans and the tile tuner report
it, and its results on batches that it does take: ids and distance bits equal
those of the per-query scan (explicit CTA layout) and of the oracle."""
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


def _layout(R, G, k, nprobe, nq, **kw):
    plan = R.Plan(G, k, nprobe, nq, **kw)
    layout = plan.tile()["layout"]
    plan.free()
    return layout


def _check(R, G, Q, k, nprobe, bq=4, eps0=1.9, **kw):
    """The batch is scanned by bucket, with the per-query scan's results."""
    import torch
    assert _layout(R, G, k, nprobe, len(Q), bq=bq, eps0=eps0) == "bucket-major"
    qd = torch.from_numpy(Q).cuda()
    ids, dist = G.search(qd, k, nprobe, bq=bq, eps0=eps0, **kw)
    ref_i, ref_d = G.search(qd, k, nprobe, bq=bq, eps0=eps0, layout=R.LAYOUT_CTA,
                            staging=R.STAGING_OFF, **kw)
    assert torch.equal(ids, ref_i)
    assert torch.equal(dist.view(torch.int32), ref_d.view(torch.int32))
    return ids.cpu().numpy(), dist.cpu().numpy()


# code lengths: one operand stage, a half stage, several, the 16-pair items of
# the longest; d below the code length (padding)
@pytest.mark.parametrize("d,bits", [(50, 64), (128, 128), (100, 192), (256, 256), (300, 320),
                                    (420, 448), (960, 1024), (2000, 2048), (4000, 4096)])
def test_code_lengths(R, d, bits):
    rng = np.random.default_rng(bits)
    n = 40_000 if bits <= 192 else 12_000 if d <= 512 else 4000
    data, Q = _mix(rng, n, d), _mix(rng, 2000, d)
    G = R.Index.build(data, 24, seed=2, code_bits=bits, kmeans_iters=3)
    for k, nprobe, eps0 in ((10, 5, 0.0), (100, 7, 1.9), (1, 24, 0.5)):
        _check(R, G, Q, k, nprobe, eps0=eps0)


@pytest.mark.parametrize("metric", ["l2", "ip", "cosine"])
@pytest.mark.parametrize("bq", [1, 3, 4])
def test_metrics_and_bits(R, metric, bq):
    rng = np.random.default_rng(7)
    data, Q = _mix(rng, 40_000, 128), _mix(rng, 2003, 128)
    G = R.Index.build(data, 32, seed=2, kmeans_iters=3, metric=metric)
    for k, nprobe in ((1, 9), (20, 9), (256, 32)):
        _check(R, G, Q, k, nprobe, bq=bq)
    _check(R, G, Q, 20, 9, bq=bq, eps0=0.0)


# one bucket of many tiles and items; buckets of 40 codes and few pairs; fewer
# codes probed than k (pads); 6000 identical points, whose upper bounds outgrow
# their list (4096 for k <= 32) while the candidates fit theirs
@pytest.mark.parametrize("n,nq,K,nprobe,k,same", [(20_000, 1031, 1, 1, 100, 0),
                                                  (40_000, 4001, 1000, 40, 10, 0),
                                                  (400, 70_001, 4, 2, 256, 0),
                                                  (12_000, 2000, 2, 1, 10, 6000)])
def test_edges_match_the_oracle(R, oracle_mod, n, nq, K, nprobe, k, same):
    from paper_2405_12497_gb300 import synth
    data, Q = synth.tiny(n=n, nq=nq)
    if same:
        data[:same] = data[0]
    G = R.Index.build(data, K, seed=2, kmeans_iters=3)
    ids, dist = _check(R, G, Q, k, nprobe)
    O = oracle_mod.OracleIndex(data, K=K, seed=2, iters=3)
    ids_o, dist_o = O.search(Q[:60], k, nprobe)
    assert np.array_equal(ids[:60], ids_o)
    assert np.array_equal(dist[:60].view(np.uint32), dist_o.view(np.uint32))


# more queries than one batch's lists hold (11570 at a share of 32768 entries):
# the second batch's offsets into the probe lists, counts and query norms
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_two_batches(R, metric):
    import torch
    rng = np.random.default_rng(9)
    data, Q = _mix(rng, 40_000, 64), _mix(rng, 12_001, 64)
    G = R.Index.build(data, 8, seed=2, kmeans_iters=3, metric=metric)
    _check(R, G, Q, 100, 8)
    npq = torch.from_numpy(rng.integers(1, 9, len(Q)).astype(np.int32)).cuda()
    _check(R, G, Q, 100, 8, per_query_nprobe=npq)


@pytest.mark.parametrize("rot", ["ROT_TF32", "ROT_BF16"])
def test_plan_rotates_beside_the_selection(R, rot):
    """A plan runs the rotation on a second stream."""
    import torch
    rng = np.random.default_rng(11)
    data, Q = _mix(rng, 40_000, 128), torch.from_numpy(_mix(rng, 2000, 128)).cuda()
    G = R.Index.build(data, 32, seed=2, kmeans_iters=3)
    plan = R.Plan(G, 50, 9, 2000, rot_precision=getattr(R, rot))
    assert plan.tile()["layout"] == "bucket-major"
    want = G.search(Q, 50, 9, rot_precision=getattr(R, rot), layout=R.LAYOUT_CTA)
    for _ in range(3):
        ids, dist = plan.search(Q)
        assert torch.equal(ids, want[0])
        assert torch.equal(dist.view(torch.int32), want[1].view(torch.int32))


def test_plans_and_the_tuner_name_the_scan(R):
    import torch
    rng = np.random.default_rng(13)
    data, Q = _mix(rng, 60_000, 128), torch.from_numpy(_mix(rng, 4000, 128)).cuda()
    G = R.Index.build(data, 64, seed=2, kmeans_iters=3)
    want = G.search(Q, 10, 16, layout=R.LAYOUT_CTA)
    assert _layout(R, G, 10, 16, 4000) == "bucket-major"
    assert _layout(R, G, 10, 16, 100) != "bucket-major"
    assert _layout(R, G, 10, 16, 4000, layout=R.LAYOUT_CTA) == "cta-per-query"
    # tuned with a small batch: the scan was not a candidate and is kept for
    # large ones, whatever staging or path was the fastest
    best, every = G.autotune_tiles(Q[:64], 10, 16, reps=2)
    assert all(t["layout"] != "bucket-major" for t in every)
    assert _layout(R, G, 10, 16, 4000) == "bucket-major"
    assert _layout(R, G, 10, 16, 100) != "bucket-major"
    # tuned with a large one: timed (0.3 of the per-query times), chosen, taken
    best, every = G.autotune_tiles(Q, 10, 16, reps=2)
    assert [t["layout"] for t in every].count("bucket-major") == 1
    assert best["layout"] == "bucket-major" and best["scan_path"] == "popcount"
    assert _layout(R, G, 10, 16, 4000) == "bucket-major"
    assert _layout(R, G, 10, 16, 100) != "bucket-major"
    ids, dist = G.search(Q, 10, 16)
    assert torch.equal(ids, want[0])
    assert torch.equal(dist.view(torch.int32), want[1].view(torch.int32))


# a learned plan selects a large batch in two parts on two streams; queries of
# few codes take their candidates from the first threshold, and a few probe
# every bucket
@pytest.mark.parametrize("nq,nprobe_max", [(4095, 48), (4099, 48), (6001, 200)])
def test_learned_plans(R, nq, nprobe_max):
    import torch
    rng = np.random.default_rng(17)
    data, Q = _mix(rng, 60_000, 128), torch.from_numpy(_mix(rng, nq, 128)).cuda()
    G = R.Index.build(data, 200, seed=2, kmeans_iters=3)
    pr = R.Predictor.train(G, torch.from_numpy(_mix(rng, 2048, 128)).cuda(), k=100,
                           nprobe_max=nprobe_max, epochs=2, batch=512)
    npq = G.predict_nprobe(pr, Q)
    plan = R.Plan(G, 100, 0, nq, predictor=pr)
    assert plan.tile()["layout"] == "bucket-major"
    want = G.search(Q, 100, nprobe_max, per_query_nprobe=npq, layout=R.LAYOUT_CTA,
                    staging=R.STAGING_OFF)
    for ids, dist in (G.search_learned(pr, Q, 100), plan.search(Q), plan.search(Q)):
        assert torch.equal(ids, want[0])
        assert torch.equal(dist.view(torch.int32), want[1].view(torch.int32))
    assert torch.equal(plan.nprobe[:nq], npq)


# squared distances down to FP32's smallest numbers
@pytest.mark.parametrize("scale", [1e-18, 1e-20, 3e-21, 1e-22])
def test_tiny_values(R, oracle_mod, scale):
    rng = np.random.default_rng(5)
    data = (_mix(rng, 20_000, 64) * scale).astype(np.float32)
    Q = (_mix(rng, 2000, 64) * scale).astype(np.float32)
    G = R.Index.build(data, 8, seed=2, kmeans_iters=2)
    O = oracle_mod.OracleIndex(data, K=8, seed=2, iters=2)
    for k, nprobe, eps0 in ((10, 4, 0.0), (10, 8, 0.5), (100, 8, 1.9)):
        ids, dist = _check(R, G, Q, k, nprobe, eps0=eps0)
        ids_o, dist_o = O.search(Q[:50], k, nprobe, eps0=eps0)
        assert np.array_equal(ids[:50], ids_o)
        assert np.array_equal(dist[:50].view(np.uint32), dist_o.view(np.uint32))
