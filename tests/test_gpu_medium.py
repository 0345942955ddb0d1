"""Medium segments at the edges of the batched sort's tiles (a segment in one
stage, in both, tile by tile with a ragged last tile) at every distance from a
16-byte boundary, for every key and value width, with constant and all-255
digits.  The oracle is numpy's stable argsort per segment (a stable sort has one
result, so equality is exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402
from paper_2607_05302_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

TILES = {(4, True): 8192, (4, False): 16384, (8, True): 6144, (8, False): 8192}


@pytest.mark.parametrize("kb,vals", sorted(TILES))
@pytest.mark.parametrize("dist", ["uniform", "low", "ones"])
def test_medium_edges(kb, vals, dist):
    t = TILES[kb, vals]
    lens = []
    for base in (4097, t, 2 * t, 3 * t, 5 * t + 777):
        for d in (-4, -3, -1, 0, 1, 2):
            lens += [max(base + d, 4097), 1 + (d & 3)]  # short ones move the next start
    off = np.zeros(len(lens) + 1, np.uint64)
    off[1:] = np.cumsum(np.array(lens, np.uint64))
    n = int(off[-1])
    r = W.splitmix64_np(kb * 7 + vals, 0, n)
    keys = (r >> np.uint64(32)).astype(np.uint32) if kb == 4 else r
    if dist == "low":
        keys &= keys.dtype.type(0xFF00FF)
    elif dist == "ones":
        keys[::2] = ~keys.dtype.type(0)
    want_k, want_v = np.empty_like(keys), np.empty(n, np.int32)
    for a, b in zip(off[:-1].astype(int), off[1:].astype(int)):
        o = np.argsort(keys[a:b], kind="stable")
        want_k[a:b] = keys[a:b][o]
        want_v[a:b] = a + o
    kt = torch.from_numpy(keys.view(np.int32 if kb == 4 else np.int64).copy()).cuda()
    vt = torch.arange(n, dtype=torch.int32, device="cuda") if vals else None
    R.sort_segmented_tensors(kt, vt, torch.from_numpy(off.view(np.int64)).cuda(), off)
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(keys.dtype), want_k)
    if vals:
        assert np.array_equal(vt.cpu().numpy(), want_v)
