"""The choice of kernel and launch geometry (host only, no GPU)."""
import numpy as np
import pytest

from paper_2309_08864_gb300 import so2dr
from tests import dispatch

RK = [(1, 1), (1, 2), (1, 3), (1, 4), (2, 1), (2, 2), (3, 1), (3, 2), (4, 1), (4, 2)]


@pytest.mark.parametrize("nx", [24, 21])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("r,k", RK)
def test_star_kernel_and_its_geometry_go_together(r, k, dtype, nx):
    """Planes of so many rows that the star kernel's tiles exceed the grid's y
    limit go to the generic kernel, not to the star kernel with the generic
    kernel's tile, grid and shared memory."""
    own = dispatch.launch(dtype, "star", r, k, (200, 4096, nx))
    assert own["fast"] == dispatch.STAR3D and not own["small"]
    limit = 65535 * own["ty"]  # rows the star kernel's grid reaches
    at = dispatch.launch(dtype, "star", r, k, (200, limit, nx))
    assert at["fast"] == dispatch.STAR3D and at["gy"] == 65535
    over = dispatch.launch(dtype, "star", r, k, (200, limit + 1, nx))
    assert not over["ok"] or over["fast"] == dispatch.GENERIC
    assert not over["ok"] or over["gy"] * over["ty"] > limit


@pytest.mark.parametrize("dtype,r,k", [("f32", 1, 4), ("f32", 4, 1), ("bf16", 1, 3)])
def test_zero_copy_only_where_the_star_kernel_runs(dtype, r, k):
    """The mapped host planes are read by the star kernel alone: plans whose
    launches its grid or its 32-bit indices cannot take have no zero-copy form
    (the generic kernel would read planes that nobody filled)."""
    c = np.full(1 + 6 * r, 1.0 / (1 + 6 * r))

    def zc(*dims):
        p = so2dr.Plan(dims, r, "star", c, k, min_chunks=2, k_on=k, k_off=k, budget_bytes=0, dtype=dtype)
        n, runs_on = p.info["zero_copy"], dispatch.launch(dtype, "star", r, k, dims)
        p.close()
        return n, runs_on["fast"] == dispatch.STAR3D and not runs_on["ragged"]

    rows = 65535 * dispatch.launch(dtype, "star", r, k, (64, 4096, 24))["ty"]
    for dims in [(64, 40, 24), (64, 40, 20), (64, 40, 21), (64, rows, 24), (64, rows + 1, 24), (64, 9, 1 << 30),
                 (64, 9, (1 << 30) + 8)]:
        has, runs_on = zc(*dims)
        assert has == runs_on, dims
    assert zc(64, 40, 24)[0] and not zc(64, rows + 1, 24)[0] and not zc(64, 9, (1 << 30) + 8)[0]


@pytest.mark.parametrize("kind,r,k", [(kind, r, 1) for kind in ("star", "box") for r in (1, 2, 3, 4)] + [("box", 4, 2), ("star", 3, 2)])
def test_short_fp64_launches_take_the_tile(kind, r, k):
    """Chunk launches of wide halos in FP64: the strips' segments stream
    mostly halo there and were slower than the generic kernel."""
    for dims, nout in [((599, 3882), 75), ((140, 2112), 140), ((64, 1000), 64), ((20, 3882), 20), ((250, 6000), 250),
                       ((12800, 12800), 300 if k == 1 else 200)]:
        assert dispatch.launch("f64", kind, r, k, dims, nout)["fast"] == dispatch.TILE2D
    if r >= 3 and k == 2:  # ragged rows, staged element by element
        assert dispatch.launch("f64", kind, r, k, (2001, 5003))["fast"] == dispatch.TILE2D
    large = dispatch.launch("f64", kind, r, k, (12800, 12800))
    assert large["fast"] == (dispatch.TILE2D if k == 1 and (kind, r) != ("box", 2) else dispatch.ROW2D)


@pytest.mark.parametrize("dims,r,k,small", [
    ((120, 129, 16), 1, 3, 0), ((185, 154, 16), 1, 4, 0), ((24, 512, 24), 1, 3, 0), ((2000, 20, 24), 1, 2, 0),
    ((600, 40, 24), 1, 3, 0), ((185, 154, 16), 3, 1, 0), ((128, 128, 128), 1, 4, 0),
    ((48, 80, 132), 1, 4, 1), ((64, 64, 64), 1, 4, 1), ((64, 64, 64), 1, 2, 1), ((60, 200, 32), 1, 2, 1),
    ((6, 352, 400), 1, 4, 1), ((64, 64, 64), 3, 1, 1), ((140, 200, 33), 1, 3, 1)])
def test_two_row_tile_only_where_its_segments_stay_short(dims, r, k, small):
    """The 2-row tile cuts a plane into more tiles and so the planes into
    fewer segments: narrow rows and long grids are the 4-row tile's."""
    assert dispatch.launch("f32", "star", r, k, dims)["small"] == small


@pytest.mark.parametrize("kind,r,k,dims", [("varcoef", 1, 2, (38, 39, 32)), ("varcoef", 1, 2, (4, 256, 256)),
                                           ("varcoef", 1, 4, (8, 256, 256)), ("star", 1, 1, (48, 48, 48)),
                                           ("star", 2, 1, (10, 512, 512)), ("star", 2, 2, (48, 48, 48)),
                                           ("star", 4, 1, (48, 48, 48))])
def test_small_fp64_plane_launches_fill_the_device(kind, r, k, dims):
    """A launch too small to occupy the SMs with the tile of least halo (38 x
    39 x 32, two levels: one tile, a few segments) gets smaller tiles; the
    tile still covers the grid and fits the shared memory."""
    sh = dispatch.launch("f64", kind, r, k, dims)
    large = dispatch.launch("f64", kind, r, k, (4000,) + dims[1:])  # the grid's tile
    assert sh["fast"] == large["fast"] == dispatch.PLANE3D
    assert sh["tx"] * sh["ty"] < large["tx"] * large["ty"]
    assert sh["gx"] * sh["tx"] >= dims[2] and sh["gy"] * sh["ty"] >= dims[1] and sh["smem"] <= 227 << 10
    assert 1 <= sh["gz"] <= dims[0]
    assert dispatch.launch("f32", "varcoef", 1, 2, dims)["tx"] == dispatch.launch("f32", "varcoef", 1, 2, (4000,) + dims[1:])["tx"]


@pytest.mark.parametrize("kind,r,k,dims", [("box", 1, 4, (600, 12800)), ("box", 2, 1, (1000, 8192)), ("star", 1, 4, (600, 12800)),
                                           ("star", 2, 2, (1000, 8192)), ("box", 1, 2, (1000, 8192))])
def test_fp64_strips_are_split_into_ctas_that_share_the_sms_evenly(kind, r, k, dims):
    """A few CTAs less than the SMs hold evenly double up on some of them."""
    sh = dispatch.launch("f64", kind, r, k, dims, occ=3)
    assert sh["fast"] == dispatch.ROW2D and sh["gx"] >= 0.93 * 152 * -(-sh["gx"] // 152)


def test_radius_two_registers_follow_the_ctas_of_the_launch():
    """One level of radius 2: registers for three CTAs per SM only where the
    launch has more than two."""
    for dims, small in [((256, 256, 256), 1), ((194, 164, 16), 1), ((20, 400, 1000), 0), ((459, 300, 728), 0), ((256, 256, 255), 0)]:
        assert dispatch.star_split_small("f32", 2, 1, dims) == small, dims
    for r, k in RK:
        assert (r, k) == (2, 1) or dispatch.star_split_small("f32", r, k, (256, 256, 256)) == 0
