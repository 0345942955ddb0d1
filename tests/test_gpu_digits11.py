"""11-bit digits in the grid layout and out of place at the edges of tiles and
blocks: a part of the rounds (every digit in two passes), all of them and the
permuted representation (rounds one by one, a truncation between them).  The
last digit of a key is narrower than the others, and keys whose digits are all
ones sit among the others (the last tile's missing elements are ranked as such
a digit).  The oracle is numpy's stable argsort of the key's low bits: a stable
sort has one result, so equality is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402
from paper_2607_05302_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

# elements of a tile, by (key bytes, values): default, with blocks of 4096
TILES = {(4, True): (10240, 8192), (4, False): (16384, 16384), (8, True): (6144, 4096), (8, False): (10240, 8192)}


def make(n, kb, seed):
    keys = W.splitmix64_np(seed, 0, n)
    keys = (keys >> np.uint64(32)).astype(np.uint32) if kb == 4 else keys
    keys[::7] = ~keys.dtype.type(0)
    keys[3::11] &= keys.dtype.type(0x00FF00FF)
    return keys


def low_bits_order(keys, bits):
    width = 8 * keys.dtype.itemsize
    low = keys if bits >= width else keys & keys.dtype.type((1 << bits) - 1)
    return np.argsort(low, kind="stable")


def to_gpu(keys, vals):
    kt = torch.from_numpy(keys.view(np.int32 if keys.dtype.itemsize == 4 else np.int64)).cuda()
    return kt, torch.arange(keys.size, dtype=torch.int32, device="cuda") if vals else None


def check(kt, vt, keys, order):
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(keys.dtype), keys[order])
    if vt is not None:
        assert np.array_equal(vt.cpu().numpy(), order.astype(np.int32))


@pytest.mark.parametrize("kb,vals", sorted(TILES))
@pytest.mark.parametrize("b", [256, 4096])
@pytest.mark.parametrize("tiles,extra", [(1, -1), (1, 0), (1, 1), (170, 5)])
def test_rounds(kb, vals, b, tiles, extra):
    n = tiles * TILES[kb, vals][b == 4096] + extra
    keys = make(n, kb, 1000 * kb + tiles + extra)
    nt = (8 * kb + 10) // 11
    for rounds in {1, 2, nt - 1, nt}:
        kt, vt = to_gpu(keys, vals)
        ko, vo = torch.empty_like(kt), torch.empty_like(vt) if vals else None
        R.sort_rounds_tensors(kt, vt, rounds, ko, vo, digit_bits=11, block_size=b, layout="grid")
        check(ko, vo, keys, low_bits_order(keys, 11 * rounds))


@pytest.mark.parametrize("kb,vals", sorted(TILES))
@pytest.mark.parametrize("how", ["grid", "grid4096", "oop", "perm"])
@pytest.mark.parametrize("tiles,extra", [(1, 1), (2, -1), (170, 5)])
def test_whole(kb, vals, how, tiles, extra):
    n = tiles * TILES[kb, vals][how == "grid4096"] + extra
    keys = make(n, kb, 2000 * kb + tiles + extra)
    nt = (8 * kb + 10) // 11
    kt, vt = to_gpu(keys, vals)
    order = low_bits_order(keys, 8 * kb)
    if how == "oop":
        R.lsd_oop_tensors(kt, vt, torch.empty_like(kt), torch.empty_like(vt) if vals else None, digit_bits=11)
    elif how == "perm":
        p = R.Perm(kt, vt, digit_bits=11, block_size=256)
        for r in range(nt):
            p.rounds(r, 1)
        m = n - n // 3
        p.truncate(m)   # the smallest m elements, then sorted again by a middle digit
        p.rounds(1, 1)
        p.finalize()
        kept = order[:m]
        mid = (keys[kept] >> keys.dtype.type(11)) & keys.dtype.type(2047)
        order = kept[np.argsort(mid, kind="stable")]
        kt, vt = kt[:m], vt[:m] if vals else None
    else:
        R.sort_tensors(kt, vt, digit_bits=11, layout="grid", block_size=4096 if how == "grid4096" else 256)
    check(kt, vt, keys, order)
