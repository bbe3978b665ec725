"""The searches, builds and trainings whose speed is measured, as a user's program runs them.

Inputs are drawn on the device from the seed alone, with the shapes and value
distributions of this repository's workloads (SIFT-, DEEP- and GIST-shaped
mixtures). A search case's index is built from centroids made here by plain
torch, so that the exact k nearest neighbours inside the probed buckets can be
computed independently in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2405_12497_gb300 import rabitq

ROT = {"fp32": rabitq.ROT_FP32, "tf32": rabitq.ROT_TF32, "bf16": rabitq.ROT_BF16}
METRICS = ("l2", "ip", "cosine")


def listed():
    return [
        # One user, one query: the smallest call there is, where launches, allocations
        # and the final wait count and not the scan.
        {"name": "one-query", "kind": "search", "data": "sift", "n": 1_000_000, "d": 128,
         "bits": 128, "K": 4096, "metric": "l2", "rot": "fp32", "host": False,
         "nq": 1, "k": 10, "nprobe": 32},
        # A serving request: a small odd batch through a search plan with learned probe
        # counts, host buffers in and out.
        {"name": "serving-request", "kind": "plan", "data": "sift", "n": 400_000, "d": 128,
         "bits": 128, "K": 2048, "metric": "l2", "rot": "fp32", "host": True,
         "nq": 53, "k": 10, "nprobe": 0, "train_nq": 2048, "nprobe_max": 256},
        # The headline workload: a 10k-query batch at recall@100 of about 0.95 through a
        # captured plan, everything resident on the device.
        {"name": "sift-batch", "kind": "plan", "data": "sift", "n": 1_000_000, "d": 128,
         "bits": 128, "K": 4096, "metric": "l2", "rot": "fp32", "host": False,
         "nq": 10_000, "k": 100, "nprobe": 62},
        # The ten nearest at a low probe count: what a recommender or a first-stage
        # retriever asks, from device memory.
        {"name": "sift-top10", "kind": "search", "data": "sift", "n": 1_000_000, "d": 128,
         "bits": 128, "K": 4096, "metric": "l2", "rot": "fp32", "host": False,
         "nq": 4_000, "k": 10, "nprobe": 16},
        # High recall on 256-dimensional unit vectors: many probes, codes far beyond the
        # caches of a small index.
        {"name": "deep-scan", "kind": "search", "data": "deep", "n": 2_000_000, "d": 256,
         "bits": 256, "K": 4096, "metric": "l2", "rot": "fp32", "host": False,
         "nq": 10_000, "k": 100, "nprobe": 128},
        # The learned probe count on a mid-sized batch: features, network, uneven counts.
        {"name": "deep-learned", "kind": "search", "data": "deep", "n": 1_000_000, "d": 256,
         "bits": 256, "K": 4096, "metric": "l2", "rot": "fp32", "host": False,
         "nq": 4_096, "k": 100, "nprobe": 0, "train_nq": 2048, "nprobe_max": 256},
        # Long vectors: 960 dimensions in 1024-bit codes with the TF32 query rotation.
        {"name": "gist-batch", "kind": "search", "data": "gist", "n": 200_000, "d": 960,
         "bits": 1024, "K": 1024, "metric": "l2", "rot": "tf32", "host": False,
         "nq": 1_000, "k": 100, "nprobe": 32},
        # Inner products over embeddings of a size that is no power of two, from host
        # arrays, an odd batch.
        {"name": "embeddings-ip", "kind": "search", "data": "deep", "n": 300_000, "d": 300,
         "bits": 320, "K": 1024, "metric": "ip", "rot": "fp32", "host": True,
         "nq": 777, "k": 50, "nprobe": 40},
        # Single-code estimates: what a graph traversal asks for scattered ids.
        {"name": "estimates", "kind": "estimate", "data": "gist", "n": 200_000, "d": 420,
         "bits": 448, "K": 1024, "metric": "l2", "rot": "fp32", "host": False,
         "nq": 1_000, "m": 128},
        # Building an index: k-means on every point, codes, factors, buckets.
        {"name": "build-sift", "kind": "build", "data": "sift", "n": 400_000, "d": 128,
         "bits": 128, "K": 2048, "metric": "l2", "iters": 10},
        # Building over long vectors: the 1024-dimensional rotation counts most.
        {"name": "build-gist", "kind": "build", "data": "gist", "n": 50_000, "d": 960,
         "bits": 1024, "K": 512, "metric": "l2", "iters": 5},
        # Training the probe-count network: labels by search, forward, backward, Adam,
        # calibration.
        {"name": "train-probes", "kind": "train", "data": "sift", "n": 300_000, "d": 128,
         "bits": 128, "K": 1024, "metric": "l2", "train_nq": 10_000, "nprobe_max": 128,
         "k": 100, "epochs": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    kind = rng.choice(["search"] * 6 + ["plan"] * 3 + ["estimate", "build", "train"])
    data = rng.choice(["sift", "sift", "deep", "deep", "gist"])
    d = {"sift": lambda: rng.choice([96, 100, 128, 128, 128, 192]),
         "deep": lambda: rng.choice([96, 200, 256, 256, 300, 384]),
         "gist": lambda: rng.choice([420, 512, 784, 960])}[data]()
    bits = (d + 63) // 64 * 64
    if d == 960:
        bits = 1024
    n = _log_int(rng, 50_000, 1_000_000 if d <= 256 else 200_000)
    K = 1 << int(round(math.log2(n / rng.uniform(100, 500))))
    metric = rng.choice(["l2", "l2", "l2", "ip", "cosine"])
    case = {"kind": kind, "data": data, "n": n, "d": d, "bits": bits, "K": K, "metric": metric,
            "rot": rng.choice(["fp32", "fp32", "tf32", "bf16"]), "host": rng.random() < 0.3}
    if kind in ("search", "plan"):
        case["nq"] = _log_int(rng, 1, 10_000 if d <= 256 else 1_500)
        case["k"] = rng.choice([1, 10, 10, 20, 50, 100, 100, 100, 150])
        case["nprobe"] = min(K, _log_int(rng, 4, 128 if d <= 256 else 64))
        if metric == "l2" and rng.random() < 0.3:
            case.update(nprobe=0, train_nq=2048, nprobe_max=min(K, 256))
    elif kind == "estimate":
        case["nq"] = _log_int(rng, 10, 2_000)
        case["m"] = rng.choice([16, 32, 64, 100, 128])
    elif kind == "build":
        case = {"kind": kind, "data": data, "n": min(n, 400_000 if d <= 256 else 60_000), "d": d,
                "bits": bits, "K": min(K, 2048 if d <= 256 else 512), "metric": metric,
                "iters": rng.choice([2, 5, 10])}
    else:
        case = {"kind": kind, "data": data, "n": min(n, 300_000), "d": d, "bits": bits,
                "K": min(K, 1024), "metric": "l2", "train_nq": _log_int(rng, 2_000, 10_000 if d <= 256 else 4_000),
                "nprobe_max": 64 if d > 256 else 128, "k": rng.choice([10, 50, 100]),
                "epochs": rng.choice([2, 5, 10])}
    return case


# ----------------------------------------------------------------- inputs

def _mixture(case, seed):
    """draw(m, stream) -> m vectors of the case's mixture, on the device."""
    kind, d, n = case["data"], case["d"], case["n"]
    dev = torch.device("cuda")

    def gen(stream):
        g = torch.Generator(device=dev)
        g.manual_seed(int(seed) * 1009 + stream)
        return g

    g = gen(0)
    if kind == "gist":
        comps = 500
        u = torch.rand((7, comps, d), generator=g, device=dev).clamp_(min=1e-30).log_().neg_()
        a, b = u[:2].sum(0), u[2:].sum(0)  # Gamma(2), Gamma(5)
        mu, spread = a / (a + b), 0.05
    elif kind == "sift":
        comps = max(10, n // 100)
        scale = torch.exp(0.5 * torch.randn(d, generator=g, device=dev))
        e = torch.rand((comps, d), generator=g, device=dev).clamp_(min=1e-30).log_().neg_()
        mu, spread = 32.0 * scale * e, 24.0 * scale
    else:
        comps = max(10, n // 100)
        mu = torch.randn((comps, d), generator=g, device=dev) / math.sqrt(d)
        spread = 0.7 / math.sqrt(d)

    def vectors(m, stream):
        gg = gen(stream)
        out = torch.empty((m, d), dtype=torch.float32, device=dev)
        for s in range(0, m, 1 << 19):
            e = min(m, s + (1 << 19))
            comp = torch.randint(0, comps, (e - s,), generator=gg, device=dev)
            x = mu[comp] + spread * torch.randn((e - s, d), generator=gg, device=dev)
            if kind == "gist":
                x = x.clamp_(0.0, 1.0)
            elif kind == "sift":
                x = x.round_().clamp_(0.0, 255.0)
            elif case["metric"] == "l2":
                x = x / x.norm(dim=1, keepdim=True)
            out[s:e] = x
        return out

    return vectors


def _nearest(x, cen):
    """Row-wise nearest centroid, in the precision of x."""
    c2 = (cen * cen).sum(1)
    out = torch.empty(x.shape[0], dtype=torch.int64, device=x.device)
    for s in range(0, x.shape[0], 1 << 15):
        out[s:s + (1 << 15)] = (c2 - 2.0 * (x[s:s + (1 << 15)] @ cen.T)).argmin(1)
    return out


def _centroids(data, K, metric):
    """K means of a sample: two Lloyd steps from evenly spaced points. Sums are
    taken in fixed point, so the same data always give the same centroids."""
    x = data[::max(1, data.shape[0] // (32 * K))]
    if metric == "cosine":
        x = x / x.norm(dim=1, keepdim=True).clamp_(min=1e-20)
    cen = x[::x.shape[0] // K][:K].clone()
    fixed = torch.round(x.double() * 2.0**24).to(torch.int64)
    for _ in range(2):
        a = _nearest(x, cen)
        cnt = torch.bincount(a, minlength=K)
        tot = torch.zeros((K, x.shape[1]), dtype=torch.int64, device=x.device)
        tot.index_add_(0, a, fixed)
        mean = tot.double() / (cnt.clamp(min=1)[:, None] * 2.0**24)
        cen = torch.where(cnt[:, None] > 0, mean.float(), cen)
    return cen.contiguous()


def _index_inputs(case, seed):
    vectors = _mixture(case, seed)
    data = vectors(case["n"], 1)
    return vectors, data, _centroids(data, case["K"], case["metric"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "build":
        return {"case": case, "seed": seed, "data": _mixture(case, seed)(case["n"], 1)}
    vectors, data, cen = _index_inputs(case, seed)
    index = rabitq.Index.build(data, case["K"], seed=seed + 2, code_bits=case["bits"],
                               centroids=cen, metric=case["metric"])
    state = {"case": case, "index": index}
    if kind == "train":
        state["queries"] = vectors(case["train_nq"], 3)
        return state
    del data
    queries = vectors(case["nq"], 2)
    state["queries"] = queries.cpu().numpy() if case["host"] else queries
    if kind == "estimate":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed * 1009 + 5)
        ids = torch.randint(0, case["n"], (case["nq"], case["m"]), generator=g, device="cuda")
        state["ids"] = ids.cpu().numpy() if case["host"] else ids
        return state
    pred = None
    if not case["nprobe"]:
        pred = rabitq.Predictor.train(index, vectors(case["train_nq"], 3), k=case["k"],
                                      nprobe_max=case["nprobe_max"], epochs=5, batch=512)
    state["predictor"] = pred
    if kind == "plan":
        state["plan"] = rabitq.Plan(index, k=case["k"], nprobe=case["nprobe"] or case["nprobe_max"],
                                    nq_max=case["nq"], predictor=pred,
                                    rot_precision=ROT[case["rot"]])
        if case["host"]:
            pin = torch.from_numpy(state["queries"]).pin_memory()
            out = (torch.empty((case["nq"], case["k"]), dtype=torch.int64).pin_memory(),
                   torch.empty((case["nq"], case["k"]), dtype=torch.float32).pin_memory())
            state["keep"] = (pin, out)
            state["queries"] = pin.numpy()
            state["out"] = (out[0].numpy(), out[1].numpy())
        else:  # results outlive the plan, whose own buffers do not
            state["out"] = (torch.empty_like(state["plan"].ids), torch.empty_like(state["plan"].dist))
    return state


# ------------------------------------------------------------------- passes

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "build":
        index = rabitq.Index.build(state["data"], case["K"], seed=state["seed"] + 2,
                                   code_bits=case["bits"], kmeans_iters=case["iters"],
                                   metric=case["metric"])
        out = {"centroids": index.centroids(), "codes": index.codes().view(np.int64),
               "factors": index.factors(), "assign": index.assign()}
        index.free()
        return out
    if kind == "train":
        pred = rabitq.Predictor.train(state["index"], state["queries"], k=case["k"],
                                      nprobe_max=case["nprobe_max"], epochs=case["epochs"])
        info = pred.info()
        out = {"params": pred.params(), "mult": info["mult"], "s0": info["s0"],
               "train_loss": info["train_loss"], "val_loss": info["val_loss"],
               "val_mean_nprobe": info["val_mean_nprobe"]}
        pred.free()
        return out
    queries = state["queries"]
    if kind == "estimate":
        return state["index"].estimate(queries, state["ids"], rot_precision=ROT[case["rot"]])
    if kind == "plan":
        plan, nq = state["plan"], case["nq"]
        if case["host"]:
            ids, dist = plan.search(queries, out=state["out"])
        else:
            plan.queries.copy_(queries)
            plan.run(nq)
            ids, dist = state["out"]
            ids.copy_(plan.ids)
            dist.copy_(plan.dist)
    elif state["predictor"] is not None:
        ids, dist = state["index"].search_learned(state["predictor"], queries, case["k"],
                                                  rot_precision=ROT[case["rot"]])
    else:
        ids, dist = state["index"].search(queries, case["k"], case["nprobe"],
                                          rot_precision=ROT[case["rot"]])
    return {"ids": ids, "dist": dist}


def work(case):
    """Each input read and each output written once; multiply-adds as two."""
    n, d, bits, K = case["n"], case["d"], case["bits"], case["K"]
    index = n * (bits / 8 + 16)
    if case["kind"] == "build":
        flops = 2.0 * n * K * d * (case["iters"] + 1) + 2.0 * n * d * bits + 4.0 * bits**3
        return {"bytes": n * d * 4 + K * d * 4 + index + n * 4, "flops": flops}
    if case["kind"] == "train":
        nq, params = case["train_nq"], 64 * 256 + 256 * 256 + 256
        pairs = nq * case["nprobe_max"] * n / K
        flops = 2.0 * nq * K * d + 2.0 * bits * pairs + 6.0 * nq * params * case["epochs"]
        return {"bytes": nq * d * 4 + K * d * 4 + index + min(n, nq * case["k"]) * d * 4 + params * 4,
                "flops": flops}
    nq = case["nq"]
    if case["kind"] == "estimate":
        pairs = nq * case["m"]
        return {"bytes": nq * d * 4 + pairs * (8 + 12 + bits / 8 + 16) + min(K, pairs) * (bits + d) * 4,
                "flops": 2.0 * nq * d * bits + pairs * 2.0 * (bits + d)}
    k = case["k"]
    probes = case["nprobe"] or case["nprobe_max"] / 4  # learned counts are well below their limit
    pairs = nq * probes * n / K
    return {"bytes": nq * d * 4 + K * d * 4 + min(n, pairs) * (bits / 8 + 16)
            + min(n, nq * k) * d * 4 + nq * k * 12,
            "flops": 2.0 * nq * K * d + 2.0 * nq * d * bits + 2.0 * bits * pairs + 3.0 * d * nq * k}


# -------------------------------------------------------------- 64-bit values

def exact(case, seed):
    """The exact distances (inner products) of the k nearest points inside the
    probed buckets. None where there is no such value: ids, randomized codes and
    estimates, trained weights, learned probe counts."""
    if case["kind"] not in ("search", "plan") or not case["nprobe"]:
        return None
    if case["n"] * (case["K"] + 2 * case["nq"]) * case["d"] > 6e12:  # beyond some 15 seconds
        return None
    vectors, data, cen = _index_inputs(case, seed)
    q = vectors(case["nq"], 2).double()
    n, k, metric = case["n"], case["k"], case["metric"]
    x, c = data.double(), cen.double()
    del data
    if metric == "cosine":
        x = x / x.norm(dim=1, keepdim=True).clamp_(min=1e-300)
        q = q / q.norm(dim=1, keepdim=True).clamp_(min=1e-300)
    cluster = _nearest(x, c)
    far = math.inf
    dist = torch.full((case["nq"], k), far, dtype=torch.float64, device="cuda")
    x2 = (x * x).sum(1) if metric == "l2" else None
    for s in range(0, case["nq"], 256):
        qq = q[s:s + 256]
        qc = qq @ c.T
        score = -qc if metric != "l2" else (c * c).sum(1) - 2.0 * qc
        near = score.topk(case["nprobe"], dim=1, largest=False).indices
        probed = torch.zeros((qq.shape[0], case["K"]), dtype=torch.bool, device="cuda")
        probed.scatter_(1, near, True)
        best = torch.full((qq.shape[0], k), far, dtype=torch.float64, device="cuda")
        for p in range(0, n, 1 << 17):
            xq = qq @ x[p:p + (1 << 17)].T
            v = -xq if metric != "l2" else (x2[p:p + (1 << 17)] - 2.0 * xq + (qq * qq).sum(1)[:, None])
            v = v.masked_fill(~probed[:, cluster[p:p + (1 << 17)]], far)
            v = v.topk(min(k, v.shape[1]), dim=1, largest=False).values
            best = torch.cat([best, v], 1).topk(k, dim=1, largest=False).values
        dist[s:s + 256] = best.clamp_(min=0.0) if metric == "l2" else best
    if metric != "l2":
        dist = -dist
    return {"ids": None, "dist": dist.cpu().numpy() if case["host"] else dist}
