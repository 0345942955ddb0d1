"""Short arrays, sorted in one launch in a cluster's shared memory: the edges of
a CTA's share and of each cluster size, every key and value width, keys with
constant digits (their rounds are skipped), float32 keys with both zeros,
infinities and NaNs, and the calls' workspaces as before.  The oracle is numpy's
stable argsort (a stable sort has one result, so equality is exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402
from paper_2607_05302_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

# positions per CTA: 512 threads x 3, 7, 13, 19 elements; clusters of 2 .. 16
SIZES = (2, 31, 511, 1535, 1536, 1537, 3584, 3585, 6144, 6145, 12289, 24576, 24577, 57344, 57345, 106496, 106497,
         131073, 155648, 155649)


def make(dist, n, kb):
    r = W.splitmix64_np(n * 31 + kb, 0, n)
    keys = (r >> np.uint64(32)).astype(np.uint32) if kb == 4 else r
    if dist == "low":
        keys = keys & keys.dtype.type(0xFF00F0)
    elif dist == "same":
        keys[:] = keys[0]
    elif dist == "ones":
        keys[::3] = ~keys.dtype.type(0)
    return keys


@pytest.mark.parametrize("kb,vals,db", [(4, True, 8), (4, False, 8), (8, True, 8), (8, False, 8), (4, True, 11)])
@pytest.mark.parametrize("dist", ["uniform", "low", "same", "ones"])
def test_small(kb, vals, db, dist):
    for n in SIZES:
        keys = make(dist, n, kb)
        order = np.argsort(keys, kind="stable")
        kt = torch.from_numpy(keys.view(np.int32 if kb == 4 else np.int64).copy()).cuda()
        vt = torch.arange(n, dtype=torch.int32, device="cuda") if vals else None
        ws = None
        if n % 2:
            ws = torch.empty(R.radsort_workspace_size(n, kb, 4 if vals else 0, db), dtype=torch.uint8, device="cuda")
        R.sort_tensors(kt, vt, digit_bits=db, workspace=ws)
        R.radsort_device_status()
        assert np.array_equal(kt.cpu().numpy().view(keys.dtype), keys[order]), n
        if vals:
            assert np.array_equal(vt.cpu().numpy(), order.astype(np.int32)), n


@pytest.mark.parametrize("n", [1000, 20_000, 100_003])
def test_float_order(n):
    bits = W.uniform_keys(n, 32, seed=n)
    bits[:8] = (0, 0x80000000, 0x7F800000, 0xFF800000, 0x7FC00000, 0xFFC00001, 1, 0x80000001)
    rank = np.where(bits >> 31, ~bits, bits ^ np.uint32(0x80000000))  # the documented total order
    order = np.argsort(rank, kind="stable")
    kt = torch.from_numpy(bits.view(np.float32).copy()).cuda()
    vt = torch.arange(n, dtype=torch.int32, device="cuda")
    R.sort_tensors(kt, vt, float_keys=True)
    R.radsort_device_status()
    assert np.array_equal(kt.view(torch.int32).cpu().numpy().view(np.uint32), bits[order])
    assert np.array_equal(vt.cpu().numpy(), order.astype(np.int32))


def test_workspace_checks():
    kt = torch.zeros(1000, dtype=torch.int32, device="cuda")
    ws = torch.empty(R.radsort_workspace_size(1000, 4, 0, 8) - 1, dtype=torch.uint8, device="cuda")
    with pytest.raises(R.RadsortError):
        R.sort_tensors(kt, workspace=ws)


def test_capture():
    keys = make("uniform", 50_000, 4)
    kt = torch.from_numpy(keys.view(np.int32).copy()).cuda()
    R.sort_tensors(kt.clone())
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        R.sort_tensors(kt)
    g.replay()
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(np.uint32), np.sort(keys))
