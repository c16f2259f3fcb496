"""The 3D star kernel's 4-row tile where small launches take the 2-row one:
grids above a million cells, and small ones with the work split pinned (which
keeps the 4-row tile), ragged and aligned rows, against the generic kernel,
bit for bit.  Each case asserts which tile it runs."""
import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import dispatch
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu

CASES = [(1, 2, "f32"), (1, 3, "f32"), (1, 4, "f32"), (3, 1, "f32"), (1, 4, "bf16"), (1, 2, "f16"), (3, 1, "bf16")]


def _same_bytes(dims, r, k, name, modes, monkeypatch):
    import torch
    dtype = so2dr.DTYPES[name]
    st = inputs.to_storage(inputs.draw_box(3, dims), dtype)
    runs = []
    for env, mode in [(None, m) for m in modes] + [("1", 1)]:
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        plan = so2dr.Plan(dims, r, "star", _coeffs(3, r, "star"), 2 * k + 1, k_on=k, k_off=k + 1, min_chunks=3,
                          budget_bytes=0, dtype=name)
        t = gu.pinned_from_storage(st.copy(), dtype)
        plan.run(t, in_core=mode)
        runs.append(t.view(torch.uint8))
        plan.close()
    for m, t in zip(modes, runs):
        assert torch.equal(t, runs[-1]), "mode %d differs from the generic kernel" % m


# odd rows, rows of even length that are no whole vectors, aligned rows; a long grid of narrow rows
@pytest.mark.parametrize("dims", [(70, 121, 125), (41, 190, 134), (41, 97, 264), (2000, 20, 24)])
@pytest.mark.parametrize("r,k,name", CASES)
def test_large_launches_match_generic_kernel_bitwise(r, k, name, dims, monkeypatch):
    sh = dispatch.launch(name, "star", r, k, dims)
    assert sh["fast"] == dispatch.STAR3D and not sh["small"]
    assert sh["ragged"] == (dims[2] % (4 if name == "f32" else 8) != 0)
    _same_bytes(dims, r, k, name, (1,), monkeypatch)


@pytest.mark.parametrize("split", ["grid", "rounds"])
@pytest.mark.parametrize("dims", [(40, 37, 121), (33, 61, 250), (26, 20, 365)])
@pytest.mark.parametrize("r,k,name", CASES)
def test_pinned_splits_on_ragged_rows_match_generic_kernel_bitwise(r, k, name, dims, split, monkeypatch):
    monkeypatch.setenv("SO2DR_WORK_SPLIT", split)
    sh = dispatch.launch(name, "star", r, k, dims)
    assert sh["fast"] == dispatch.STAR3D and sh["ragged"] and not sh["small"]
    _same_bytes(dims, r, k, name, (1, 0), monkeypatch)
