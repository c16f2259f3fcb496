"""The two 2D kernels on either side of the rule that picks one: strips on
launches of many rows, the shared-memory tile on short ones, against the
generic kernel, bit for bit."""
import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1100, 1500), (700, 2051), (9, 33), (300, 515)])
@pytest.mark.parametrize("kind,r,k,name", [("box", 1, 8, "f32"), ("box", 2, 3, "f32"), ("box", 4, 1, "f32"),
                                           ("box", 4, 2, "f16"), ("star", 1, 4, "f32"), ("star", 3, 4, "bf16"),
                                           ("star", 1, 4, "f64"), ("star", 2, 3, "f64"), ("box", 2, 2, "f64"),
                                           ("star", 2, 1, "f64")])
def test_strips_and_tiles_match_generic_kernel_bitwise(kind, r, k, name, dims, monkeypatch):
    import torch
    dtype = so2dr.DTYPES[name]
    if min(dims) <= 2 * r:
        pytest.skip("no interior")
    st = inputs.to_storage(inputs.draw_box(3, dims), dtype)
    runs = []
    for env, mode in ((None, 1), (None, 0), ("1", 1)):
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        plan = so2dr.Plan(dims, r, kind, _coeffs(2, r, kind), 2 * k + 1, k_on=k, k_off=k + 1, min_chunks=1,
                          budget_bytes=0, dtype=name)
        t = gu.pinned_from_storage(st.copy(), dtype)
        plan.run(t, in_core=mode)
        runs.append(t.view(torch.uint8))
        plan.close()
    assert torch.equal(runs[0], runs[2]), "in-core differs from the generic kernel"
    assert torch.equal(runs[1], runs[2]), "out-of-core differs from the generic kernel"
