"""The batched sort at the limits of its workspace.  A few medium segments are
sorted with the long ones where that takes at most 1 MiB more; a caller whose
workspace holds the plan without that, but not the 1 MiB, gets that plan (the
in-place plans can need far more: 304 CTAs' blocks where there are many short
medium segments).  The sizes are asked for without a GPU."""
import ctypes

import numpy as np
import pytest

from paper_2607_05302_gb300 import radsort as R

LENS = [65_536] * 8 + [16_000] * 560  # 9.5M elements: 6% of them is under 16 of the longest


def offsets(lens):
    off = np.zeros(len(lens) + 1, np.uint64)
    off[1:] = np.cumsum(np.array(lens, np.uint64))
    return off


def plain(off, kb, vb):
    """The fastest plan without a group: the counters, two lists and the
    alternate arrays of 16 CTAs."""
    def up(x):
        return (x + 255) // 256 * 256

    lens = np.diff(off.astype(np.int64))
    nseg, per = len(lens), 16 * int(lens.max())
    return 256 + 2 * up(nseg * 4) + up(per * kb) + (up(per * 4) if vb else 0)


@pytest.mark.parametrize("kb,vb", [(4, 4), (8, 4), (8, 0)])
def test_smallest_workspace(kb, vb):
    off = offsets(LENS)
    p = plain(off, kb, vb)
    most = R.segmented_workspace_size(off, kb, vb)
    assert p < most <= p + (1 << 20)  # the group is worth its memory here
    assert R.segmented_workspace_size(off, kb, vb, minimal=True) == p


@pytest.mark.gpu
@pytest.mark.parametrize("kb", [4, 8])
@pytest.mark.parametrize("extra", [0, 1, -1])
def test_sort_in_it(kb, extra):
    torch = pytest.importorskip("torch")
    from test_gpu_groups import batch

    off, keys, want_k, want_v = batch(LENS, kb, 31)
    size = R.segmented_workspace_size(off, kb, 4, minimal=True) if extra < 1 else \
        R.segmented_workspace_size(off, kb, 4) - 1
    kt = torch.from_numpy(keys.view(np.int32 if kb == 4 else np.int64).copy()).cuda()
    vt = torch.arange(keys.size, dtype=torch.int32, device="cuda")
    od = torch.from_numpy(off.view(np.int64)).cuda()
    ws = torch.empty(size + (256 if extra < 0 else 0), dtype=torch.uint8, device="cuda")
    if extra < 0:  # one byte short
        oh = np.ascontiguousarray(off)
        got = R.lib().radsort_sort_segmented(ctypes.c_void_p(kt.data_ptr()), ctypes.c_void_p(vt.data_ptr()),
                                             ctypes.c_void_p(od.data_ptr()), oh.ctypes.data_as(ctypes.c_void_p),
                                             len(LENS), kb, 8, ctypes.c_void_p(ws.data_ptr()), size - 1, None)
        assert got == R.RADSORT_ENOMEM
        return
    R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(keys.dtype), want_k)
    assert np.array_equal(vt.cpu().numpy(), want_v)
