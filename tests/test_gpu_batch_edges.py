"""The batched sort at the edges of its plan, each form told by its launches:
medium segments of several tiles on one CTA each (u32 keys alone have the longest
tiles), the line where a few medium segments are grouped, and groups at the limit
of 64 arrays.  The oracle is numpy's stable argsort per segment (a stable sort has
one result, so equality is exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402
from test_gpu_groups import batch  # noqa: E402

pytestmark = pytest.mark.gpu

PASSES = 3  # classification, short and medium segments


def group(kb):
    return 2 + kb  # counts, bucket starts, a round per byte


def check(lens, kb, vals, seed, launches):
    off, keys, want_k, want_v = batch(lens, kb, seed)
    kt = torch.from_numpy(keys.view(np.int32 if kb == 4 else np.int64).copy()).cuda()
    vt = torch.arange(keys.size, dtype=torch.int32, device="cuda") if vals else None
    od = torch.from_numpy(off.view(np.int64)).cuda()
    ws = torch.empty(R.segmented_workspace_size(off, kb, 4 if vals else 0), dtype=torch.uint8, device="cuda")
    before = R.radsort_launch_count()
    R.sort_segmented_tensors(kt, vt, od, off, workspace=ws)
    assert R.radsort_launch_count() - before == launches
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(keys.dtype), want_k)
    if vals:
        assert np.array_equal(vt.cpu().numpy(), want_v)


@pytest.mark.parametrize("d", [-3, -1, 0, 1, 2])
def test_u32_keys_tile_by_tile(d):
    t = 16384
    lens = []
    for base in (2 * t, 2 * t + 5, 3 * t, 3 * t + 777):
        lens += [base + d, 1 + (d & 3)]  # the short ones move the next start
    check(lens, 4, False, 41 + d, PASSES)


@pytest.mark.parametrize("kb,vals", [(4, True), (4, False), (8, True), (8, False)])
def test_line_of_the_few(kb, vals):
    check([65_535, 1, 40_001, 65_535], kb, vals, 51, PASSES)
    check([65_536, 1, 40_001, 65_535], kb, vals, 52, PASSES + group(kb))


@pytest.mark.parametrize("kb", [4, 8])
@pytest.mark.parametrize("num", [32, 33, 64, 65])
def test_number_of_the_few(num, kb):
    lens = [120_000] + [16_385 + 61 * i for i in range(num - 1)]
    check(lens, kb, True, 60 + num, PASSES + (group(kb) if num <= 64 else 0))


@pytest.mark.parametrize("num,groups", [(33, 1), (64, 1), (65, 2), (130, 3)])
def test_number_in_a_group(num, groups):
    # the first, unaligned, makes the four streams' slices hold 24M elements
    check([1, 6_000_000] + [262_145 + 4 * (i % 3) for i in range(num - 1)], 4, True, 70 + num, PASSES + 6 * groups)
