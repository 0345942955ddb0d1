"""float32 keys in the grid layout, where the first pass reads them as ordered
integers and the last writes them back: bit patterns with both zeros, NaN,
infinities and subnormals, and digits that are constant in the first pass, the
last, both or all (such a pass is left out, and a pass over the array takes
its place), with tails of every kind.  The oracle is numpy's stable argsort of
the ordered integers; bit-exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402

pytestmark = pytest.mark.gpu


def make(kind, n):
    rng = np.random.default_rng(n + len(kind))
    bits = rng.integers(0, 2 ** 32, n, dtype=np.uint64).astype(np.uint32)
    special = np.array([0, 0x80000000, 0x7F800000, 0xFF800000, 0x7FC00001, 0xFFC00001, 1, 0x80000001], np.uint32)
    if kind == "bits":
        bits[::5] = special[np.arange(bits[::5].size) % special.size]
    if kind in ("first", "both"):  # the lowest byte is constant
        bits &= np.uint32(0x7FFFFF00)
    if kind in ("last", "both"):   # the highest one is
        bits = (bits & np.uint32(0x00FFFFFF)) | np.uint32(0xC0000000)
    if kind == "first":            # (negative ones would have another lowest byte)
        bits[::3] |= np.uint32(0x00800000)
    if kind == "equal":
        bits[:] = 0xBF812345
    return bits


@pytest.mark.parametrize("kind", ["bits", "first", "last", "both", "equal"])
@pytest.mark.parametrize("vals", [True, False])
@pytest.mark.parametrize("n", [200_000, 10240 * 23, 16384 * 17 + 1, 1_000_003])
@pytest.mark.parametrize("plan", [dict(block_size=64), dict(block_size=2048), dict(block_size=512, shape=2),
                                  dict(block_size=4096, digit_bits=11)])
def test_passes(kind, vals, n, plan):
    bits = make(kind, n)
    kt = torch.from_numpy(bits.view(np.float32).copy()).cuda()
    vt = torch.arange(n, dtype=torch.int32, device="cuda") if vals else None
    R.sort_tensors(kt, vt, float_keys=True, layout="grid", **plan)
    R.radsort_device_status()
    ordered = np.where(bits >> 31, ~bits, bits | np.uint32(0x80000000))
    order = np.argsort(ordered, kind="stable")
    assert np.array_equal(kt.view(torch.int32).cpu().numpy().view(np.uint32), bits[order])
    if vals:
        assert np.array_equal(vt.cpu().numpy(), order.astype(np.int32))
