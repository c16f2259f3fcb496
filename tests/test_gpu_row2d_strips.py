"""The 2D strip kernel at every (R, K) it is built for, on launches long
enough that the shared-memory tile does not take them: tall grids of few
columns and wide ones of few rows (a strip exactly, one column more or less,
rows that are no whole vectors, fewer rows than the fused halo), and grids
whose strips are cut into long segments and a tail of short ones.  Against the
generic kernel, bit for bit; each case asserts the kernel and the split it runs."""
import functools

import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import dispatch
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu

BOX = [(1, k) for k in range(1, 9)] + [(2, 1), (2, 2), (2, 3), (2, 4), (3, 1), (3, 2), (3, 3), (4, 1), (4, 2)]
STAR = [(1, k) for k in range(1, 9)] + [(r, k) for r in (2, 3, 4) for k in (1, 2, 3, 4)]
WIDE = [(1, 1), (1, 2), (1, 3), (1, 4), (2, 1), (2, 2), (2, 3), (2, 4), (3, 1), (3, 2), (4, 1), (4, 2)]  # FP64
CASES = [("box", r, k, "f32") for r, k in BOX] + [("star", r, k, "f32") for r, k in STAR]
CASES += [(kind, r, k, "f64") for kind in ("box", "star") for r, k in WIDE if k > 1 or (kind, r) == ("box", 2)]
CASES += [("box", 1, 8, "bf16"), ("box", 3, 2, "bf16"), ("box", 4, 1, "f16"), ("star", 2, 4, "f16"),
          ("star", 1, 4, "bf16"), ("star", 4, 3, "bf16")]


@functools.lru_cache(maxsize=4)
def _grid(dims, dtype):
    return inputs.to_storage(inputs.draw_box(3, dims), dtype)


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _same_bytes(dims, kind, r, k, name, modes, monkeypatch):
    import torch
    dtype = so2dr.DTYPES[name]
    st = _grid(dims, dtype)
    runs = []
    for env, mode in [(None, m) for m in modes] + [("1", 1)]:
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        # a launch of depth k and one single step
        plan = so2dr.Plan(dims, r, kind, _coeffs(2, r, kind), k + 1, k_on=k, k_off=k + 1, min_chunks=3,
                          budget_bytes=0, dtype=name)
        t = gu.pinned_from_storage(st.copy(), dtype)
        plan.run(t, in_core=mode)
        runs.append(t.view(torch.uint8))
        plan.close()
    for m, t in zip(modes, runs):
        assert torch.equal(t, runs[-1]), "mode %d differs from the generic kernel" % m


@pytest.mark.parametrize("dims", [(156000, 20), (156000, 29), (39000, 124), (39000, 125), (31300, 149), (12100, 411),
                                  (17, 294000), (17, 294001)])
@pytest.mark.parametrize("kind,r,k,name", CASES)
def test_strips_match_generic_kernel_bitwise(kind, r, k, name, dims, monkeypatch):
    if name == "f64" and r > 2 and dims[1] % 4:  # the tile takes these up to twice as many rows
        dims = (dims[0] * 9 // 4, dims[1])
    sh = dispatch.launch(name, kind, r, k, dims, sms=_sms())
    wide = kind == "box" and (r, k) == (2, 4) and name != "f64" and dims[1] % 4 == 0
    assert sh["fast"] == (dispatch.BOX2D if wide else dispatch.ROW2D)
    _same_bytes(dims, kind, r, k, name, (1,), monkeypatch)


@pytest.mark.parametrize("dims", [(270000, 20), (180001, 125)])
@pytest.mark.parametrize("kind,r,k,name", [("box", 1, 8, "f32"), ("box", 1, 1, "f32"), ("box", 4, 2, "f32"),
                                           ("box", 2, 3, "bf16"), ("box", 2, 2, "f64"), ("star", 1, 8, "f32"),
                                           ("star", 3, 4, "f32"), ("star", 1, 4, "f16"), ("star", 2, 4, "f64"),
                                           ("star", 4, 2, "f64")])
def test_long_and_short_segments_match_generic_kernel_bitwise(kind, r, k, name, dims, monkeypatch):
    for occ in range(1, 5):  # whatever number of CTAs fits an SM
        sh = dispatch.launch(name, kind, r, k, dims, sms=_sms(), occ=occ)
        assert sh["fast"] == dispatch.ROW2D and sh["split2"] > 0 and 0 < sh["split_at"] < dims[0]
    _same_bytes(dims, kind, r, k, name, (1, 0), monkeypatch)


@pytest.mark.parametrize("dims", [(75, 3882), (64, 1000), (33, 125), (20, 31), (900, 5003)])
@pytest.mark.parametrize("kind,r,k", [(kind, r, 1) for kind in ("star", "box") for r in (1, 2, 3, 4)] + [("box", 4, 2), ("star", 3, 2)])
def test_fp64_tile_matches_generic_kernel_bitwise(kind, r, k, dims, monkeypatch):
    assert dispatch.launch("f64", kind, r, k, dims, sms=_sms())["fast"] == dispatch.TILE2D
    _same_bytes(dims, kind, r, k, "f64", (1, 0), monkeypatch)
