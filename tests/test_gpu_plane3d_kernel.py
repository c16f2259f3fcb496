"""The plane-streaming 3D kernel (FP64 stars, the variable-coefficient star)
against the generic kernel, bit for bit, in core and out of core: tiles of one
and two column groups, ragged rows, grids smaller than a tile, fused depths
whose halo leaves few rows."""
import numpy as np
import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import dispatch
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(30, 21, 33), (41, 66, 57), (19, 70, 130), (28, 13, 9)])
@pytest.mark.parametrize("kind,r,k,name", [("star", 1, 1, "f64"), ("star", 1, 4, "f64"), ("star", 2, 2, "f64"),
                                           ("star", 3, 2, "f64"), ("star", 4, 1, "f64"), ("star", 4, 2, "f64"),
                                           ("varcoef", 1, 1, "f32"), ("varcoef", 1, 4, "f32"),
                                           ("varcoef", 1, 6, "f32"), ("varcoef", 1, 3, "f64")])
def test_plane_kernel_matches_generic_kernel_bitwise(kind, r, k, name, dims, monkeypatch):
    _same_bytes(kind, r, k, name, dims, monkeypatch)


# the tile of a large FP64 launch, and ones fitted to few and to thin planes
@pytest.mark.parametrize("dims", [(61, 230, 231), (13, 301, 257), (70, 40, 61)])
@pytest.mark.parametrize("kind,r,k", [("star", 1, 4), ("star", 2, 2), ("star", 4, 1), ("varcoef", 1, 3)])
def test_large_and_fitted_fp64_tiles_match_generic_kernel_bitwise(kind, r, k, dims, monkeypatch):
    grid_tile = dispatch.launch("f64", kind, r, k, (4000,) + dims[1:])
    own = dispatch.launch("f64", kind, r, k, dims)
    if dims[0] == 61:
        assert (own["tx"], own["ty"]) == (grid_tile["tx"], grid_tile["ty"])
    _same_bytes(kind, r, k, "f64", dims, monkeypatch)


def _same_bytes(kind, r, k, name, dims, monkeypatch):
    import torch
    dtype = so2dr.DTYPES[name]
    st = inputs.to_storage(inputs.draw_box(3, dims), dtype)
    cf = None
    if kind == "varcoef":
        cf = torch.from_numpy(np.stack([inputs.draw_box(100 + f, dims, a=0.05, b=0.15) for f in range(6)]).astype(st.dtype)).pin_memory()
    runs = []
    for env, mode in ((None, 1), (None, 0), ("1", 1)):
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        plan = so2dr.Plan(dims, r, kind, None if cf is not None else _coeffs(3, r, "star"), 2 * k + 1, k_on=k,
                          k_off=k + 1, min_chunks=3, budget_bytes=0, dtype=name)
        t = gu.pinned_from_storage(st.copy(), dtype)
        plan.run(t, cf, in_core=mode)
        runs.append(t)
        plan.close()
    assert torch.equal(runs[0], runs[2]), "in-core differs from the generic kernel"
    assert torch.equal(runs[1], runs[2]), "out-of-core differs from the generic kernel"
