"""With little device memory left a large batch falls back to the per-query
scan's smaller scratch, whichever allocation it is that does not fit. Runs in a
process of its own: the rest of the device's memory is taken by a tensor."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = """
import ctypes
import torch
from paper_2405_12497_gb300 import rabitq as R

rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])

def room():
    # give the stream-ordered pool's memory back, then the bytes free
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    pool = ctypes.c_void_p()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert rt.cudaMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
    return torch.cuda.mem_get_info()[0]

def leave(nbytes):
    return torch.empty(room() - nbytes, dtype=torch.uint8, device="cuda")

g = torch.Generator(device="cuda")
g.manual_seed(1)
data = torch.randn((200_000, 64), generator=g, device="cuda")
MB = 1 << 20
"""


def _run(code):
    r = subprocess.run([sys.executable, "-c", COMMON + code], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    return r.stdout


# the lists of 2000 queries take about 1 GB, the per-query kernel's 640 MB
def test_search_with_little_memory():
    out = _run("""
G = R.Index.build(data, 64, seed=2, kmeans_iters=2)
Q = torch.randn((2000, 64), generator=g, device="cuda")
want = G.search(Q, 100, 16, layout=R.LAYOUT_CTA)
G.search(Q, 100, 16)
for mb in (2600, 1900, 1650, 1400, 1200, 1000, 850):
    held = leave(mb * MB)
    got = G.search(Q, 100, 16)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]), mb
    del held
print("ok")
""")
    assert "ok" in out


def test_plan_with_little_memory():
    out = _run("""
G = R.Index.build(data, 64, seed=2, kmeans_iters=2)
nq = 200_000
Q = torch.randn((nq, 64), generator=g, device="cuda")
before = room()
plan = R.Plan(G, 100, 16, nq)
need = before - room()
plan.search(Q[:1100])
plan.free()
small = R.Plan(G, 100, 16, nq, layout=R.LAYOUT_CTA)
want = small.search(Q[:1100].cpu().numpy())
small.free()
# short of the last buffer, of the last two, of all three, of the scratch
for less in (20, 100, 180, 300, 1000):
    held = leave(need - less * MB)
    p = R.Plan(G, 100, 16, nq)
    del held
    torch.cuda.empty_cache()
    got = p.search(Q[:1100].cpu().numpy())
    assert (got[0] == want[0]).all() and (got[1] == want[1]).all(), less
    p.free()
print("ok")
""")
    assert "ok" in out


# the assignment's tiles and lists take 1 GB here, the rows' 8-bit copy 0.4 GB:
# a build that fits without them fits with any more memory, too
def test_build_with_little_memory():
    out = _run("""
n, K = 4_000_000, 64
data = torch.randn((n, 64), generator=g, device="cuda")
want = R.Index.build(data, K, seed=2, kmeans_iters=2)
cen, codes = want.centroids(), want.codes()
want.free()
fits = []
for mb in range(1100, 3300, 100):
    held = leave(mb * MB)
    try:
        G = R.Index.build(data, K, seed=2, kmeans_iters=2)
    except R.RabitqError as e:
        assert e.code == -2, e
        fits.append(False)
    else:
        fits.append(True)
        if len(fits) % 5 == 0:
            assert (G.centroids() == cen).all() and (G.codes() == codes).all(), mb
        G.free()
    del held
print("".join(".x"[f] for f in fits))
assert fits[-1] and fits == sorted(fits), fits
print("ok")
""")
    assert "ok" in out
