"""The tensor-core k-means assignment (kernels_assign.cu) against the oracle's
scan of all canonical distances: centroid bits and assignments are equal.
The products only choose what is scored canonically, so nothing is tolerated."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2405_12497_gb300 import rabitq
    return rabitq


def _check(R, oracle_mod, data, K, iters, **kw):
    G = R.Index.build(data, K, seed=5, kmeans_iters=iters, **kw)
    cent, assign, _ = oracle_mod.kmeans(data, K, iters, 5, threads=os.cpu_count() or 1)
    assert np.array_equal(G.centroids().view(np.uint32), cent.view(np.uint32))
    assert np.array_equal(G.assign(), assign)


# the smallest rows and centroids that take it, ragged row blocks and column
# tiles, K steps of one to several MMAs and several stages, one dimension
@pytest.mark.parametrize("n,d,K", [(4096, 64, 64), (4097, 65, 257), (5000, 96, 255), (4100, 1, 64),
                                   (4223, 17, 300), (9000, 130, 513), (4096, 960, 100),
                                   (4500, 2050, 70), (60000, 24, 1025)])
def test_sizes(R, oracle_mod, n, d, K):
    rng = np.random.default_rng(n + d)
    _check(R, oracle_mod, rng.standard_normal((n, d)).astype(np.float32), K, 2)


# ties and duplicates (lists overflow: rows scanned canonically), all rows
# equal, a far offset, scales outside the scaled range, overflowing distances
@pytest.mark.parametrize("what", ["integers", "duplicates", "equal", "offset", "tiny", "small",
                                  "large", "overflow", "mixed"])
def test_values(R, oracle_mod, what):
    rng = np.random.default_rng(3)
    x = rng.standard_normal((6000, 40)).astype(np.float32)
    if what == "integers":
        x = rng.integers(0, 2, x.shape).astype(np.float32)
    elif what == "duplicates":
        x = np.repeat(x[:30], 200, axis=0)
    elif what == "equal":
        x[:] = x[0]
    elif what == "offset":
        x = 3e4 + x
    elif what == "tiny":
        x *= np.float32(1e-19)
    elif what == "small":
        x *= np.float32(1e-14)
    elif what == "large":
        x *= np.float32(1e17)
    elif what == "overflow":
        x[::7] *= np.float32(1e25)
    elif what == "mixed":
        x[::3] *= np.float32(1e-9)
        x[1::3] *= np.float32(1e6)
    _check(R, oracle_mod, x, 100, 1)


def test_device_rows_at_any_address(R, oracle_mod):
    """Rows of a device array that starts 4 bytes past an aligned address."""
    import torch
    rng = np.random.default_rng(8)
    data = rng.standard_normal((4200, 32)).astype(np.float32)
    flat = torch.zeros(4200 * 32 + 1, device="cuda")
    flat[1:] = torch.from_numpy(data).reshape(-1).cuda()
    G = R.Index.build(flat[1:].view(4200, 32), 80, seed=5, kmeans_iters=2)
    cent, assign, _ = oracle_mod.kmeans(data, 80, 2, 5, threads=4)
    assert np.array_equal(G.centroids().view(np.uint32), cent.view(np.uint32))
    assert np.array_equal(G.assign(), assign)


def test_row_chunks(R):
    """More rows than a GiB of operand tiles holds (8388608 at up to 64
    dimensions): the rows at the chunks' ends are assigned as in builds of
    their own, small enough for the canonical scan."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    chunk, d, K = 1 << 23, 16, 70
    cen = torch.randn((K, d), generator=g, device="cuda")
    n = chunk + 5001
    data = cen[torch.randint(0, K, (n,), generator=g, device="cuda")]
    data += 0.5 * torch.randn((n, d), generator=g, device="cuda")
    G = R.Index.build(data, K, seed=2, centroids=cen)
    got = G.assign()
    for at in (0, chunk - 4000, chunk, n - 4000):
        S = R.Index.build(data[at:at + 4000].contiguous(), K, seed=2, centroids=cen)
        assert np.array_equal(got[at:at + 4000], S.assign()), at
        S.free()
    G.free()
