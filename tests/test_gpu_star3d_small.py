"""The 3D star kernel's two tile heights on either side of the rule that picks
one (a million cells): the same bytes as the generic kernel, through the
device-resident entry point."""
import ctypes

import pytest

from paper_2309_08864_gb300 import inputs, so2dr
from tests import gpu_util as gu
from tests.test_gpu_parity import _coeffs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(48, 80, 132), (9, 11, 13), (25, 33, 31), (110, 97, 100), (61, 12, 24)])
@pytest.mark.parametrize("r,k,name", [(1, 2, "f32"), (1, 3, "f32"), (1, 4, "f32"), (3, 1, "f32"), (1, 4, "bf16"),
                                      (1, 3, "f16"), (3, 1, "bf16")])
def test_both_tile_heights_match_generic_kernel_bitwise(r, k, name, dims, monkeypatch):
    import torch
    dtype, T = so2dr.DTYPES[name], 2 * k + 1
    c = list(_coeffs(3, r, "star"))
    src = gu.pinned_from_storage(inputs.to_storage(inputs.draw_box(3, dims), dtype), dtype).cuda()
    lib = so2dr.load_library()
    outs = []
    for env in (None, "1"):
        if env:
            monkeypatch.setenv("SO2DR_GENERIC_KERNEL", env)
        dst = torch.empty_like(src)
        rc = lib.so2dr_run_device_noalloc(3, (ctypes.c_int64 * 3)(*dims), r, so2dr.STAR, (ctypes.c_double * len(c))(*c),
                                          len(c), T, k, dtype, ctypes.c_void_p(src.data_ptr()),
                                          ctypes.c_void_p(dst.data_ptr()),
                                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == so2dr.OK, lib.so2dr_last_error().decode()
        torch.cuda.synchronize()
        outs.append(dst.cpu().view(torch.uint8))
    assert torch.equal(outs[0], outs[1])
