"""CTAs per SM of the 3D star kernel at one level: its plane loop waits for
copies, and a resident CTA less cost radius 2 up to a fifth of its speed."""
import pytest

from tests import dispatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("r,ctas", [(1, 3), (2, 3), (4, 2)])
def test_one_level_occupancy(r, ctas, dtype):
    assert dispatch.star_occupancy(dtype, r, 1, (64, 256, 256)) >= ctas
