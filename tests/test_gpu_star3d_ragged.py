"""The 3D star kernel on rows that are no whole 16-byte units (staged element
by element) against the generic kernel, bit for bit: in core and out of core,
rows shorter than a tile, one column around a tile's edge, the right ring
straddling two lanes, odd and even 16-bit rows."""
import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu

RK = [(1, 1), (1, 2), (1, 3), (1, 4), (2, 1), (2, 2), (3, 1), (3, 2), (4, 1), (4, 2)]
CASES = [(r, k, so2dr.F32, "f32") for r, k in RK]
CASES += [(1, 4, so2dr.BF16, "bf16"), (2, 1, so2dr.BF16, "bf16"), (1, 3, so2dr.F16, "f16"), (4, 1, so2dr.F16, "f16")]


@pytest.mark.parametrize("dims", [(40, 37, 121), (33, 61, 250), (57, 26, 43), (30, 70, 127), (26, 20, 365)])
@pytest.mark.parametrize("r,k,dtype,name", CASES)
def test_ragged_rows_match_generic_kernel_bitwise(r, k, dtype, name, dims, monkeypatch):
    import torch
    st = inputs.to_storage(inputs.draw_box(3, dims), dtype)
    runs = []
    for env, mode in ((None, 1), (None, 0), ("1", 1)):
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        plan = so2dr.Plan(dims, r, "star", _coeffs(3, r, "star"), 2 * k + 1, k_on=k, k_off=k + 1, min_chunks=3,
                          budget_bytes=0, dtype=name)
        t = gu.pinned_from_storage(st.copy(), dtype)
        plan.run(t, in_core=mode)
        runs.append(t.view(torch.uint8))
        plan.close()
    assert torch.equal(runs[0], runs[2]), "in-core differs from the generic kernel"
    assert torch.equal(runs[1], runs[2]), "out-of-core differs from the generic kernel"
