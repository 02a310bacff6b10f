"""GPU rotated BEV NMS (rtcc_nms) against the oracle's float64 IoU and greedy
rule, on constructed box sets: ragged and full 32-box chunks, the largest
list (512), duplicates, disjoint sets, suppression chains, and thresholds 0
and 1."""
import concurrent.futures as cf
import math
import os
import subprocess
import sys

import numpy as np
import pytest

from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    return U.load()


def _boxes(rows):
    b = np.zeros(len(rows), dtype=U.R.BOX_DTYPE)
    for i, (x, y, l, w, yaw) in enumerate(rows):
        b[i] = (x, y, -1.0, l, w, 1.5, yaw, 1.0 - i * 1e-3, i)
    return b


def _crowd(n, seed, spread=12.0):
    """n car-sized boxes around a few centres, so many pairs overlap."""
    rng = np.random.default_rng(seed)
    centres = rng.uniform(-spread, spread, size=(max(1, n // 24), 2))
    c = centres[rng.integers(0, len(centres), n)]
    xy = c + rng.normal(scale=1.0, size=(n, 2))
    l = 3.9 * np.exp(rng.normal(scale=0.2, size=n))
    w = 1.6 * np.exp(rng.normal(scale=0.2, size=n))
    yaw = rng.choice([0.0, math.pi / 2], n) + rng.normal(scale=0.3, size=n)
    return _boxes(np.column_stack([xy[:, 0], xy[:, 1], l, w, yaw]))


@pytest.mark.parametrize("n,seed", [(1, 0), (31, 1), (32, 2), (33, 3), (200, 4), (512, 5)])
@pytest.mark.parametrize("thr", [0.15, 0.5])
def test_nms_crowded_sets(R, n, seed, thr):
    b = _crowd(n, seed)
    out = R.rtcc_nms(b, thr)
    kept = U.check_nms(b, out, thr)
    assert kept[0] == 0
    if n >= 200:
        assert len(kept) < n                           # the crowd does overlap


def test_nms_edge_cases(R):
    assert len(R.rtcc_nms(np.zeros(0, dtype=R.BOX_DTYPE), 0.15)) == 0
    same = _boxes([(5.0, -3.0, 3.9, 1.6, 0.4)] * 40)
    same["anchor"] = np.arange(40)
    assert R.rtcc_nms(same, 0.15)["anchor"].tolist() == [0]
    far = _boxes([(10.0 * i, 0.0, 3.9, 1.6, 0.1 * i) for i in range(64)])
    assert R.rtcc_nms(far, 0.0)["anchor"].tolist() == list(range(64))
    # A-B and B-C at IoU 1/2, A-C at 1/5: B falls to A, C survives
    chain = _boxes([(0.0, 0.0, 1.0, 1.0, 0.0), (1 / 3, 0.0, 1.0, 1.0, 0.0), (2 / 3, 0.0, 1.0, 1.0, 0.0)])
    assert R.rtcc_nms(chain, 0.3)["anchor"].tolist() == [0, 2]
    assert R.rtcc_nms(chain, 0.1)["anchor"].tolist() == [0]
    crowd = _crowd(128, 9)
    assert R.rtcc_nms(crowd, 1.0)["anchor"].tolist() == list(range(128))
    out = R.rtcc_nms(crowd, 0.0)                         # any overlap suppresses
    U.check_nms(crowd, out, 0.0)


def test_nms_threads_and_shrinking_lists(R):
    """Calls from more threads than workspaces stay allocated, each with lists
    of changing length: every call sees its own boxes only."""
    lists = [_crowd(n, 40 + i) for i, n in enumerate([512, 1, 65, 300, 32, 7, 511, 128])]
    want = [R.rtcc_nms(b, 0.2) for b in lists]
    for b, out in zip(lists, want):
        U.check_nms(b, out, 0.2)

    def turn(t):
        return [(i, R.rtcc_nms(lists[i], 0.2)) for r in range(12) for i in [(t + r) % len(lists)]]

    with cf.ThreadPoolExecutor(8) as ex:
        for got in ex.map(turn, range(8)):
            for i, out in got:
                assert out.tobytes() == want[i].tobytes()


@pytest.mark.parametrize("n", [64, 65, 224, 255, 256, 257, 481, 512])
def test_nms_suppressors_in_any_earlier_chunk(R, n):
    """A row of boxes that overlap their neighbours, ranked at random: what
    removes a box lies in its own 32-box chunk, the one before or any earlier
    one, in odd and even numbers of chunks, the last one full or not."""
    rng = np.random.default_rng(n)
    x = rng.permutation(n) * 1.7
    b = _boxes(np.column_stack([x, np.zeros(n), np.full(n, 4.0), np.full(n, 1.8), np.zeros(n)]))
    kept = U.check_nms(b, R.rtcc_nms(b, 0.2), 0.2)
    assert n // 4 <= len(kept) <= n // 2 + 1           # IoU 0.40 to a neighbour, 0.08 two on


CONTEXTS = """
import ctypes as C, sys
import numpy as np
from tests import gpu_util as U
from tests.test_gpu_nms import _crowd
R, cu = U.load(), C.CDLL("libcuda.so.1")
boxes = [_crowd(n, n) for n in (512, 33)]
dev, primary, cur = C.c_int(), C.c_void_p(), C.c_void_p()
def ok(r): assert r == 0, r
ok(cu.cuInit(0)); ok(cu.cuDeviceGet(C.byref(dev), 0)); ok(cu.cuDevicePrimaryCtxRetain(C.byref(primary), dev))
want = None
for turn in range(6):                       # a context of its own, then the primary one
    ctx = C.c_void_p()
    ok(cu.cuCtxCreate_v2(C.byref(ctx), C.c_uint(0), dev))
    for c in (ctx, primary, ctx):
        ok(cu.cuCtxSetCurrent(c))
        got = [R.rtcc_nms(b, 0.2).tobytes() for b in boxes]
        want = want or got
        assert got == want
        ok(cu.cuCtxGetCurrent(C.byref(cur)))
        assert cur.value == c.value
    ok(cu.cuCtxSetCurrent(primary))
    ok(cu.cuCtxDestroy_v2(ctx))
for b, g in zip(boxes, want):
    U.check_nms(b, R.rtcc_nms(b, 0.2), 0.2)
print("contexts ok")
"""


def test_nms_in_contexts_that_come_and_go(R):
    """Calls in driver contexts that are created and destroyed, and in the primary
    one between them: workspaces of a context that is gone are never used."""
    r = subprocess.run([sys.executable, "-c", CONTEXTS], cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "contexts ok" in r.stdout, r.stdout + r.stderr
