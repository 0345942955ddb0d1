"""Long segments sorted in groups (more of them than a group holds, ragged last
tiles, every distance from a 16-byte boundary, every key and value width), and
the few medium segments that join them, also under capture without a call before
it.  The oracle is numpy's stable argsort per segment (a stable sort has one
result, so equality is exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402
from paper_2607_05302_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def batch(lens, kb, seed):
    off = np.zeros(len(lens) + 1, np.uint64)
    off[1:] = np.cumsum(np.array(lens, np.uint64))
    n = int(off[-1])
    r = W.splitmix64_np(seed, 0, n)
    keys = (r >> np.uint64(32)).astype(np.uint32) if kb == 4 else r
    keys[: n // 3] &= keys.dtype.type(0xFF0FFF)
    keys[::5] = ~keys.dtype.type(0)
    want_k, want_v = np.empty_like(keys), np.empty(n, np.int32)
    for a, b in zip(off[:-1].astype(int), off[1:].astype(int)):
        o = np.argsort(keys[a:b], kind="stable")
        want_k[a:b] = keys[a:b][o]
        want_v[a:b] = a + o
    return off, keys, want_k, want_v


def check(lens, kb, vals, seed, capture=False):
    off, keys, want_k, want_v = batch(lens, kb, seed)
    kt = torch.from_numpy(keys.view(np.int32 if kb == 4 else np.int64).copy()).cuda()
    vt = torch.arange(keys.size, dtype=torch.int32, device="cuda") if vals else None
    od = torch.from_numpy(off.view(np.int64)).cuda()
    ws = torch.empty(max(1, R.segmented_workspace_size(off, kb, 4 if vals else 0)), dtype=torch.uint8, device="cuda")
    if capture:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)
        g.replay()
    else:
        R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(keys.dtype), want_k)
    if vals:
        assert np.array_equal(vt.cpu().numpy(), want_v)


def test_few_medium_captured():
    check([70_000, 5, 100_001, 20_000, 131_073, 3000], 4, True, 11, capture=True)


@pytest.mark.parametrize("kb,vals", [(4, True), (4, False), (8, True), (8, False)])
def test_few_medium(kb, vals):
    check([65_536, 1, 262_144, 2, 99_999, 3, 17_000, 16_384, 6, 30_721], kb, vals, 12)


@pytest.mark.parametrize("kb,vals", [(4, True), (4, False), (8, True), (8, False)])
def test_long(kb, vals):
    check([262_145, 1, 300_007, 2, 524_289, 3, 262_146, 5000, 1_048_577], kb, vals, 13)


def test_more_than_a_group():
    check([262_145 + 7 * i for i in range(66)] + [9000], 4, True, 14)
