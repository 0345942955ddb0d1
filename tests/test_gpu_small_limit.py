"""The longest arrays that go to the one-launch sort, by element width and by
whether the caller has given a workspace: past them a sort takes the launches of
the round kernel."""
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kb,vals,given,most", [
    (4, True, True, 155_648), (4, False, True, 155_648), (8, False, True, 155_648), (8, True, True, 57_344),
    (4, True, False, 155_648), (4, False, False, 155_648), (8, False, False, 155_648), (8, True, False, 106_496)])
def test_limit(kb, vals, given, most):
    for n in (1000, most, most + 1):
        kt = torch.arange(n, 0, -1, dtype=torch.int32 if kb == 4 else torch.int64, device="cuda")
        vt = torch.arange(n, dtype=torch.int32, device="cuda") if vals else None
        ws = torch.empty(R.radsort_workspace_size(n, kb, 4 if vals else 0, 8), dtype=torch.uint8,
                         device="cuda") if given else None
        before = R.radsort_launch_count()
        R.sort_tensors(kt, vt, workspace=ws)
        launches = R.radsort_launch_count() - before
        R.radsort_device_status()
        assert (launches == 1) == (n <= most), (n, launches)
        assert torch.equal(kt, torch.arange(1, n + 1, dtype=kt.dtype, device="cuda"))
        if vals:
            assert torch.equal(vt, torch.arange(n - 1, -1, -1, dtype=torch.int32, device="cuda"))
