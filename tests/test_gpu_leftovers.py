"""Long segments too large for the pool that the groups share, beside some that
are grouped: results, plain and captured, and that those left over are spread
over the library's streams again.  The oracle is numpy's stable argsort per
segment (a stable sort has one result, so equality is exact).  The spread is read
off the captured graph: the longest chain of dependent launches grows by the
launches of the segments on one stream, not of all of them."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402
from test_gpu_groups import batch  # noqa: E402

pytestmark = pytest.mark.gpu

STREAMS = 4  # of the plan with the full workspace


def longest_chain(graph):
    """Nodes on the longest path of a captured graph (CUgraph)."""
    drv = ctypes.CDLL("libcuda.so.1")
    num = ctypes.c_size_t(0)
    assert drv.cuGraphGetEdges(graph, None, None, ctypes.byref(num)) == 0 and num.value
    src, dst = (ctypes.c_void_p * num.value)(), (ctypes.c_void_p * num.value)()
    assert drv.cuGraphGetEdges(graph, src, dst, ctypes.byref(num)) == 0
    succ, indeg = {}, {}
    for a, b in zip(src, dst):
        succ.setdefault(a, []).append(b)
        indeg.setdefault(a, 0)
        indeg[b] = indeg.get(b, 0) + 1
    depth, todo = {x: 1 for x in indeg}, [x for x in indeg if not indeg[x]]
    while todo:
        a = todo.pop()
        for b in succ.get(a, ()):
            depth[b] = max(depth[b], depth[a] + 1)
            indeg[b] -= 1
            if not indeg[b]:
                todo.append(b)
    return max(depth.values())


def captured_chain(lens):
    """The longest chain of one call's captured graph (it is not run)."""
    drv = ctypes.CDLL("libcuda.so.1")
    off = np.zeros(len(lens) + 1, np.uint64)
    off[1:] = np.cumsum(np.array(lens, np.uint64))
    kt = torch.zeros(int(off[-1]), dtype=torch.int32, device="cuda")
    vt = torch.zeros_like(kt)
    od = torch.from_numpy(off.view(np.int64)).cuda()
    ws = torch.empty(R.segmented_workspace_size(off, 4, 4), dtype=torch.uint8, device="cuda")
    R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)  # the library's streams exist
    torch.cuda.synchronize()
    st, graph = torch.cuda.Stream(), ctypes.c_void_p(0)
    handle = ctypes.c_void_p(st.cuda_stream)
    assert drv.cuStreamBeginCapture_v2(handle, 1) == 0  # this thread's
    try:
        R.sort_segmented_tensors(kt, vt, od, off, workspace=ws, stream=st)
    finally:
        assert drv.cuStreamEndCapture(handle, ctypes.byref(graph)) == 0
    try:
        return longest_chain(graph)
    finally:
        drv.cuGraphDestroy(graph)


def test_left_over_segments_are_spread():
    alone = captured_chain([1 << 22])            # one Radsort
    grouped = captured_chain([1 << 22, 70_000])  # a group, then one
    eight = captured_chain([1 << 22] * 8 + [70_000])
    # two a stream: one more Radsort than with one, and a few nodes of the fork
    assert eight <= grouped + alone * (8 // STREAMS - 1) + 4, (alone, grouped, eight)


@pytest.mark.parametrize("kb,vals", [(4, True), (4, False), (8, True), (8, False)])
@pytest.mark.parametrize("capture", [False, True])
def test_results(kb, vals, capture):
    lens = [1 << 21] * 5 + [70_000, 3, 1 << 19, 300_001, 100_003, 5000, (1 << 20) + 8]
    off, keys, want_k, want_v = batch(lens, kb, 21)
    k0 = torch.from_numpy(keys.view(np.int32 if kb == 4 else np.int64).copy()).cuda()
    v0 = torch.arange(keys.size, dtype=torch.int32, device="cuda") if vals else None
    kt, vt = k0.clone(), v0.clone() if vals else None
    od = torch.from_numpy(off.view(np.int64)).cuda()
    ws = torch.empty(R.segmented_workspace_size(off, kb, 4 if vals else 0), dtype=torch.uint8, device="cuda")
    g = None
    if capture:
        R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)
    for _ in range(3):  # the slices are used again by the next call
        kt.copy_(k0)
        if vals:
            vt.copy_(v0)
        if capture:
            g.replay()
        else:
            R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)
        R.radsort_device_status()
        assert np.array_equal(kt.cpu().numpy().view(keys.dtype), want_k)
        if vals:
            assert np.array_equal(vt.cpu().numpy(), want_v)
