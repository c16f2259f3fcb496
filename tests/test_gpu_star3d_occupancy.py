"""CTAs per SM of the 3D star kernel at one level: its plane loop waits for
copies, and a resident CTA less cost radius 2 up to a fifth of its speed."""
import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import dispatch
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("r,ctas", [(1, 3), (2, 3), (4, 2)])
def test_one_level_occupancy(r, ctas, dtype):
    assert dispatch.star_occupancy(dtype, r, 1, (64, 256, 256)) >= ctas


@pytest.mark.parametrize("dims", [(48, 64, 96), (194, 164, 16), (64, 256, 264), (20, 400, 1000)])
@pytest.mark.parametrize("name", ["f32", "bf16", "f16"])
def test_radius_two_forms_match_generic_kernel_bitwise(name, dims, monkeypatch):
    """Radius 2 at one level, in the forms for two and for three CTAs per SM."""
    import torch
    dtype = so2dr.DTYPES[name]
    st = inputs.to_storage(inputs.draw_box(3, dims), dtype)
    runs = []
    for env, mode in ((None, 1), (None, 0), ("1", 1)):
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        plan = so2dr.Plan(dims, 2, "star", _coeffs(3, 2, "star"), 3, k_on=1, k_off=2, min_chunks=3, budget_bytes=0, dtype=name)
        t = gu.pinned_from_storage(st.copy(), dtype)
        plan.run(t, in_core=mode)
        runs.append(t.view(torch.uint8))
        plan.close()
    assert torch.equal(runs[0], runs[2]) and torch.equal(runs[1], runs[2])
