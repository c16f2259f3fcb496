"""The 2D register-streaming kernel (box and star, any row length, every
storage type) against the generic kernel, bit for bit: both sum a cell's
products in the same order and round only at kernel stores.  Sizes sit where
the strips and segments can go wrong: rows shorter than a strip, one strip
exactly, one column more or less, rows that are no whole vectors, two-column
remainders, fewer rows than the fused halo."""
import numpy as np
import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu

NAMES = {so2dr.F64: "f64", so2dr.F32: "f32", so2dr.BF16: "bf16", so2dr.F16: "f16"}
DEPTHS = {("box", "f32"): [(1, 1), (1, 8), (2, 3), (2, 4), (3, 2), (3, 3), (4, 1), (4, 2)],
          ("star", "f32"): [(1, 1), (1, 5), (1, 8), (2, 4), (3, 4), (4, 3), (4, 4)],
          ("box", "f64"): [(1, 4), (2, 3), (3, 2), (4, 2)],
          ("star", "f64"): [(1, 1), (1, 4), (2, 4), (3, 2), (4, 2)]}
CASES = [(kind, r, k, so2dr.F64 if ct == "f64" else so2dr.F32) for (kind, ct), v in DEPTHS.items() for r, k in v]
CASES += [("box", 1, 8, so2dr.BF16), ("box", 4, 1, so2dr.F16), ("star", 2, 4, so2dr.F16), ("star", 1, 4, so2dr.BF16)]


@pytest.mark.parametrize("dims", [(61, 124), (33, 125), (150, 411), (47, 20), (19, 1030), (700, 37)])
@pytest.mark.parametrize("kind,r,k,dtype", CASES)
def test_row2d_matches_generic_kernel_bitwise(kind, r, k, dtype, dims, monkeypatch):
    import torch
    st = inputs.to_storage(inputs.draw_box(3, dims), dtype)
    T = 2 * k + 1  # two launches of depth k and one single step
    runs = []
    for env, mode in ((None, 1), (None, 0), ("1", 1)):
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        plan = so2dr.Plan(dims, r, kind, _coeffs(2, r, kind), T, k_on=k, k_off=k + 1, min_chunks=3,
                          budget_bytes=0, dtype=NAMES[dtype])
        t = gu.pinned_from_storage(st.copy(), dtype)
        plan.run(t, in_core=mode)
        runs.append(t.view(torch.uint8))
        plan.close()
    assert torch.equal(runs[0], runs[2]), "in-core differs from the generic kernel"
    assert torch.equal(runs[1], runs[2]), "out-of-core differs from the generic kernel"
    assert not torch.equal(runs[0], gu.pinned_from_storage(st.copy(), dtype).view(torch.uint8))
