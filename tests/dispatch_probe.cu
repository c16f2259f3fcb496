// dispatch_probe.cu -- the library's own choice of kernel and geometry for one
// launch, for tests (host code only: no CUDA call).
#include "kernels.hpp"

using namespace so2dr;

// out: {ok, kernel family, 2-row tile, ragged, grid x, y, z, tile x, y, shared
// bytes, split, split2, split_at}; the families are LaunchShape::fast's.
extern "C" void probe_launch(int dtype, int shape, int r, int depth, int64_t n0, int64_t ny, int64_t nx, int64_t nout,
                             int sms, int occ, int64_t* out) {
    const int csize = dtype == SO2DR_F64 ? 8 : 4;
    const int esize = dtype == SO2DR_F64 ? 8 : dtype == SO2DR_F32 ? 4 : 2;
    LaunchShape ls = stencil_launch_shape(shape, r, depth, n0, ny, nx, csize, esize);
    StencilArgs a = {};
    a.split_at = nout;
    if (ls.ok && ls.fast == kFastRow2D && !tile2d_short(ls, shape, nout, nx, r, depth, csize, sms))
        choose_row_split(ls, nout, r, depth, csize, sms, occ, a);
    if (ls.ok && ls.fast == kFastPlane3D) {
        plane_fit(ls, nout, r, depth, ny, nx, csize, sms);
        ls.grid.z = (unsigned)choose_segments((int64_t)ls.grid.x * ls.grid.y, nout, r, depth, sms, 1, false);
    }
    if (ls.ok && ls.fast == kFastStar3D) star_small(ls, nout, ny, nx, r, depth, esize, sms);
    const int64_t v[13] = {ls.ok, ls.fast, ls.small, ls.ragged, ls.ok ? ls.grid.x : 0, ls.ok ? ls.grid.y : 0,
                           ls.ok ? ls.grid.z : 0, ls.ok ? ls.tx : 0, ls.ok ? ls.ty : 0, ls.ok ? (int64_t)ls.smem : 0,
                           a.split, a.split2, a.split_at};
    for (int i = 0; i < 13; ++i) out[i] = v[i];
}

// Whether a 3D star launch's split takes the form for few CTAs.
extern "C" int probe_star_split_small(int dtype, int r, int depth, int64_t n0, int64_t ny, int64_t nx, int sms, int occ) {
    LaunchShape ls = stencil_launch_shape(kStar3D, r, depth, n0, ny, nx, 4, dtype == SO2DR_F32 ? 4 : 2);
    ls.grid.z = 1;
    int split = 0;
    choose_work_split(ls, n0, r, depth, sms, occ, &split);
    return ls.small;
}

// CTAs per SM the driver reports for the 3D star kernel of a launch (needs a
// GPU); -1: another kernel.
extern "C" int probe_star_occupancy(int dtype, int r, int depth, int64_t n0, int64_t ny, int64_t nx) {
    const int esize = dtype == SO2DR_F32 ? 4 : 2;
    LaunchShape ls = stencil_launch_shape(kStar3D, r, depth, n0, ny, nx, 4, esize);
    return ls.ok && ls.fast == kFastStar3D ? stencil_occupancy(dtype, kStar3D, r, depth, ls) : -1;
}
