"""The digit width is not a matter of timing where both widths run the same
passes: 8 comes back with the plan that radsort_autotune finds for it, and
nothing more is launched than for that plan."""
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
@pytest.mark.parametrize("n", [1, 1000, R.RADSORT_SCRATCH_MAX_N, R.RADSORT_SCRATCH_MAX_N + 1, (1 << 22) + 3])
def test_same_passes(dtype, n):
    kt = torch.arange(n, 0, -1, dtype=dtype, device="cuda")
    vt = torch.arange(n, dtype=torch.int32, device="cuda")
    plan = R.radsort_autotune(kt, vt, digit_bits=8)
    before = R.radsort_launch_count()
    assert R.radsort_autotune_digits(kt, vt) == (8, *plan)
    assert R.radsort_launch_count() == before  # the plan is cached
