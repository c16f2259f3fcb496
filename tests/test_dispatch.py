"""The choice of kernel and launch geometry (host only, no GPU)."""
import pytest

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
