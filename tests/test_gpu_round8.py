"""The 8-bit round kernel at the edges of its tiles: one element short of a
tile, a tile, one past it, a ragged last tile, and more tiles than SMs, in
the grid layout (both tile shapes) and out of place.  Keys whose digits are all
255 sit among the others: the last tile's missing elements are ranked as digit
255 behind the real ones.  The oracle is numpy's stable argsort (a stable sort
has one result, so equality is exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402
from paper_2607_05302_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

# elements of a tile of the default shape, by (key bytes, values)
TILES = {(4, True): 10240, (4, False): 16384, (8, True): 6144, (8, False): 10240}


def make(n, kb, seed):
    keys = W.splitmix64_np(seed, 0, n)
    keys = (keys >> np.uint64(32)).astype(np.uint32) if kb == 4 else keys
    keys[::7] = ~keys.dtype.type(0)   # every digit 255
    keys[3::11] &= keys.dtype.type(0x00FF00FF)
    return keys


@pytest.mark.parametrize("kb,vals", sorted(TILES))
@pytest.mark.parametrize("tiles,extra", [(1, -1), (1, 0), (1, 1), (2, 17), (40, -33), (330, 5)])
@pytest.mark.parametrize("how", ["grid", "shape2", "oop"])
def test_tile_edges(kb, vals, tiles, extra, how):
    n = tiles * TILES[kb, vals] + extra
    keys = make(n, kb, 1000 * kb + tiles + extra)
    order = np.argsort(keys, kind="stable")
    kt = torch.from_numpy(keys.view(np.int32 if kb == 4 else np.int64)).cuda()
    vt = torch.arange(n, dtype=torch.int32, device="cuda") if vals else None
    if how == "oop":
        R.lsd_oop_tensors(kt, vt, torch.empty_like(kt), None if vt is None else torch.empty_like(vt))
    else:
        R.sort_tensors(kt, vt, layout="grid", block_size=256, shape=2 if how == "shape2" else 0)
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(keys.dtype), keys[order])
    if vals:
        assert np.array_equal(vt.cpu().numpy(), order.astype(np.int32))
