// kernels.cu -- launch geometry and dtype dispatch of the stencil kernel.
#include "kernels.hpp"
#include "box2d_fast.cuh"
#include "plane_tb.cuh"
#include "row2d_tb.cuh"
#include "star3d_tb.cuh"
#include "tile2d_tb.cuh"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

namespace so2dr {

namespace {
constexpr int64_t kSmemLimit = 200 * 1024;

bool is3d(int shape) { return shape == kStar3D || shape == kVarcoef3D; }

// Loaded-tile edge for an in-plane halo H: at least 32 and at least 2H + 16.
int tile_edge(int H) {
    int e = 2 * H + 16;
    if (e < 32) e = 32;
    return (e + 7) / 8 * 8;
}
}  // namespace

bool fast_star3d_supported(int r, int depth) {
    return (r == 1 && depth >= 1 && depth <= 4) || (r >= 2 && r <= 4 && depth >= 1 && depth <= 2);
}

bool fast_star3d_row_ok(int64_t nx, int esize) { return nx % (esize == 4 ? 4 : 8) == 0; }

bool fast_box2d_supported(int r, int depth) {
    return depth >= 1 && ((r == 1 && depth <= 8) || (r == 2 && depth <= 4) || (r == 3 && depth <= 3) ||
                          (r == 4 && depth <= 2));
}

// Radius 2, four levels, on 12800^2 FP32: 825 Gcell-steps/s against 730 with
// the warp strips of row2d_tb.cuh, which give 16 of their 128 columns to the
// halo there.  The other (R, K) are faster in strips (radius 1: 1763 / 1504 at
// 8 levels, 1828 / 1289 at 4; radius 2: 730 / 605 at 1, 759 / 670 at 2;
// radius 3: 481 / 368 at 1; radius 4: 321 / 246 at 1, 287 / 239 at 2), or the
// same (radius 3 at 3 levels: 403 / 404).
bool wide_box2d(int r, int depth, int64_t nx, int csize) { return r == 2 && depth == 4 && nx % 4 == 0 && csize == 4; }

bool row2d_supported(int shape, int r, int depth, int csize) {
    if (depth < 1 || r < 1 || r > 4 || (shape != kBox2D && shape != kStar2D)) return false;
    // FP64 state takes twice the registers
    if (csize == 8) return depth <= (r <= 2 ? 4 : 2);
    if (shape == kBox2D) return fast_box2d_supported(r, depth);
    return depth <= (r == 1 ? 8 : 4);
}

namespace {
// The 2D kernel's geometry; ls.grid.x is the strips until choose_row_split.
void row_shape(LaunchShape& ls, int shape, int r, int depth, int64_t nx, int csize, int esize) {
    const int kind = shape == kBox2D ? kRowBox : kRowStar;
    ls.lx = 32 * row_vx(kind, csize, r, depth);
    ls.ly = 1;
    ls.tx = ls.lx - 2 * row_hxa(r, depth);
    ls.ty = 1;
    ls.ragged = nx % 4 != 0;
    ls.block = dim3(32 * kRowWarps, 1, 1);
    ls.smem = (size_t)row_smem(kind, csize, esize, r, depth);
    ls.grid = dim3((unsigned)((nx + ls.tx - 1) / ls.tx), 1, 1);
    ls.ok = true;
    ls.fast = kFastRow2D;
}

// The plane kernel's tile: the one that computes the fewest rows of 32 cells
// over the grid (halos and the grid's last, partial tiles included; a row
// loaded counts 0.3, a phase's barrier and bookkeeping 12).  With sms > 0, for
// one launch of nout planes that cannot fill the device with such tiles: the
// least time of the busiest SM instead.  A CTA of a segment of len planes loads
// one plane a phase, len + 2H + depth phases that last 32 rows' time at least,
// and level l computes len + 2r(depth - l) planes; the given tile keeps its
// place unless another is 10% better.
void plane_shape(LaunchShape& ls, int r, int depth, int64_t ny, int64_t nx, int csize, int64_t nout = 0, int sms = 0) {
    const int H = r * depth;
    const int lx0 = ls.lx, ly0 = ls.ly;
    double best = -1;
    for (int lx : {32, 64})
        for (int ly = 2 * H + 4; ly <= kPlaneMaxRows * (kPlaneThreads / lx); ly += 4) {
            const int tx = lx - 2 * H, ty = ly - 2 * H;
            const int64_t smem = plane_smem_bytes(r, depth, lx, ly, csize);
            if (tx <= 0 || smem > kSmemLimit) continue;
            const int64_t gx = (nx + tx - 1) / tx, gy = (ny + ty - 1) / ty;
            if (gx > 2147483647 || gy > 65535) continue;
            double cost;
            if (sms > 0) {
                const int64_t tiles = gx * gy, fill = tiles < sms ? sms / tiles : 1;
                const int64_t n = std::min<int64_t>(std::min<int64_t>(fill, 64), nout);
                const double len = (double)nout / (double)n, phases = len + 2.0 * H + depth;
                double rows = phases * 0.3 * ly;
                for (int l = 1; l <= depth; ++l) rows += (len + 2.0 * r * (depth - l)) * (ly - 2 * l * r);
                cost = (double)((tiles * n + sms - 1) / sms) * (rows * (lx / 32) + phases * 32.0);
                if (lx == lx0 && ly == ly0) cost *= 0.9;
            } else {
                double rows = 0.3 * ly;
                for (int l = 1; l <= depth; ++l) rows += ly - 2 * l * r;
                cost = (double)gx * (double)gy * (rows * (lx / 32) + 12.0);
            }
            if (best >= 0 && cost >= best) continue;
            best = cost;
            ls.lx = lx;
            ls.ly = ly;
            ls.tx = tx;
            ls.ty = ty;
            ls.smem = (size_t)smem;
            ls.grid = dim3((unsigned)gx, (unsigned)gy, 1);
            ls.ok = true;
        }
    ls.block = dim3(kPlaneThreads, 1, 1);
    ls.fast = kFastPlane3D;
}

template <int R, int K, bool SMALL = false> void fast_shape(LaunchShape& ls, int64_t ny, int64_t nx, int esize) {
    using S = StarShape<R, K, SMALL>;
    ls.small = SMALL;
    ls.lx = S::LX;
    ls.ly = S::LYT;
    ls.tx = S::TX;
    ls.ty = S::TY;
    ls.block = dim3(S::NT, 1, 1);
    ls.smem = esize == 4 ? S::template smem<4>() : S::template smem<2>();
    ls.grid = dim3((unsigned)((nx + S::TX - 1) / S::TX), (unsigned)((ny + S::TY - 1) / S::TY), 1);
    ls.ragged = !fast_star3d_row_ok(nx, esize);
    if (ls.ragged) ls.smem += S::ragged_bytes;
    ls.ok = ls.grid.y <= 65535;
    ls.fast = kFastStar3D;
}
}  // namespace

LaunchShape stencil_launch_shape(int shape, int r, int depth, int64_t n0, int64_t ny, int64_t nx, int csize, int esize) {
    LaunchShape ls;
    ls.ok = false;
    ls.fast = 0;
    ls.ragged = ls.small = false;
    if (depth < 1) return ls;
    const bool fast_ok = n0 <= kMaxFastAxis && ny <= kMaxFastAxis && nx <= kMaxFastAxis &&
                         !std::getenv("SO2DR_GENERIC_KERNEL");
    if (fast_ok && shape == kBox2D && wide_box2d(r, depth, nx, csize)) {
        using S = BoxShape<2, 4>;
        ls.lx = S::LX;
        ls.ly = 1;
        ls.tx = S::TX;
        ls.ty = 1;
        ls.block = dim3(S::NT, 1, 1);
        ls.smem = esize == 4 ? S::template smem<4>() : S::template smem<2>();
        ls.grid = dim3((unsigned)((nx + S::TX - 1) / S::TX), 1, 1);
        ls.ok = true;
        ls.fast = kFastBox2D;
        return ls;
    }
    // the 2D kernel takes every other 2D launch of a depth it is built for: on
    // 16384^2 and 5003 x 6001 grids it was faster than the generic kernel at
    // every depth, radius and type
    if (fast_ok && row2d_supported(shape, r, depth, csize)) {
        row_shape(ls, shape, r, depth, nx, csize, esize);
        return ls;
    }
    if (shape == kStar3D && csize == 4 && fast_star3d_supported(r, depth) && fast_ok) {
        switch (r * 16 + depth) {
            case 17: fast_shape<1, 1>(ls, ny, nx, esize); break;
            case 18: fast_shape<1, 2>(ls, ny, nx, esize); break;
            case 19: fast_shape<1, 3>(ls, ny, nx, esize); break;
            case 20: fast_shape<1, 4>(ls, ny, nx, esize); break;
            case 33: fast_shape<2, 1>(ls, ny, nx, esize); break;
            case 34: fast_shape<2, 2>(ls, ny, nx, esize); break;
            case 49: fast_shape<3, 1>(ls, ny, nx, esize); break;
            case 50: fast_shape<3, 2>(ls, ny, nx, esize); break;
            case 65: fast_shape<4, 1>(ls, ny, nx, esize); break;
            case 66: fast_shape<4, 2>(ls, ny, nx, esize); break;
        }
        if (ls.ok) return ls;
        // more rows than the star kernel's grid reaches (65535 tiles in y): all
        // of the choice is taken back, the generic kernel has its own geometry
        ls.fast = 0;
        ls.ragged = false;
    }
    int H = r * depth;
    // (only depths the generic kernel takes too, so that the deepest supported
    // launch does not depend on the kernel)
    if (fast_ok && ny * nx <= kMaxFastAxis && (shape == kVarcoef3D || (shape == kStar3D && csize == 8)) &&
        stencil_smem_bytes(shape, r, depth, tile_edge(H), tile_edge(H), csize) <= kSmemLimit) {
        plane_shape(ls, r, depth, ny, nx, csize);
        if (ls.ok) return ls;
        ls.fast = 0;
    }
    if (is3d(shape)) {
        ls.lx = ls.ly = tile_edge(H);
        ls.tx = ls.lx - 2 * H;
        ls.ty = ls.ly - 2 * H;
        ls.block = dim3(32, 8, 1);
    } else {
        ls.lx = 256;
        while (ls.lx - 2 * H < 64) ls.lx += 128;
        ls.ly = 1;
        ls.tx = ls.lx - 2 * H;
        ls.ty = 1;
        ls.block = dim3(256, 1, 1);
    }
    ls.smem = (size_t)stencil_smem_bytes(shape, r, depth, ls.lx, ls.ly, csize);
    if ((int64_t)ls.smem > kSmemLimit) return ls;
    int64_t gx = (nx + ls.tx - 1) / ls.tx;
    int64_t gy = is3d(shape) ? (ny + ls.ty - 1) / ls.ty : 1;
    if (gx > 2147483647 || gy > 65535) return ls;
    ls.grid = dim3((unsigned)gx, (unsigned)gy, 1);
    ls.ok = true;
    return ls;
}

bool star3d_reads_host(int r, int depth, int64_t n0, int64_t ny, int64_t nx, int esize) {
    const LaunchShape ls = stencil_launch_shape(kStar3D, r, depth, n0, ny, nx, 4, esize);
    return ls.ok && ls.fast == kFastStar3D && !ls.ragged;
}

int stencil_max_depth(int shape, int r, int csize) {
    int best = 0;
    for (int d = 1; d <= 16; ++d) {
        LaunchShape ls = stencil_launch_shape(shape, r, d, 1024, 1024, 1024, csize, csize);
        if (ls.ok) best = d;
    }
    return best;
}

int stencil_occupancy(int dtype, int shape, int r, int depth, const LaunchShape& ls) {
    if (ls.fast == kFastStar3D) switch (dtype) {
        case SO2DR_F32: return ls.ragged ? occupancy_star3d_ragged_f32(r, depth, ls) : occupancy_star3d_f32(r, depth, ls);
        case SO2DR_BF16: return ls.ragged ? occupancy_star3d_ragged_bf16(r, depth, ls) : occupancy_star3d_bf16(r, depth, ls);
        case SO2DR_F16: return ls.ragged ? occupancy_star3d_ragged_f16(r, depth, ls) : occupancy_star3d_f16(r, depth, ls);
        default: return 1;
    }
    if (ls.fast == kFastRow2D) switch (dtype) {
        case SO2DR_F64: return occupancy_row2d_f64(shape, r, depth, ls);
        case SO2DR_F32: return occupancy_row2d_f32(shape, r, depth, ls);
        case SO2DR_BF16: return occupancy_row2d_bf16(shape, r, depth, ls);
        case SO2DR_F16: return occupancy_row2d_f16(shape, r, depth, ls);
        default: return 1;
    }
    switch (dtype) {
        case SO2DR_F64: return occupancy_stencil_f64(shape, r, depth, ls);
        case SO2DR_F32: return occupancy_stencil_f32(shape, r, depth, ls);
        case SO2DR_BF16: return occupancy_stencil_bf16(shape, r, depth, ls);
        case SO2DR_F16: return occupancy_stencil_f16(shape, r, depth, ls);
        default: return 1;
    }
}

int choose_segments(int64_t tiles, int64_t nout, int r, int depth, int sms, int occ, bool share_sm) {
    if (tiles <= 0 || nout <= 0 || sms <= 0) return 1;
    const int64_t slots = (int64_t)sms * (share_sm || occ < 1 ? 1 : occ);
    int best = 1;
    double best_cost = 0;
    for (int n = 1; n <= 64 && n <= nout; ++n) {
        // share_sm: the CTAs resident on one SM share its throughput, so an
        // SM's time goes with the CTAs it receives (the busiest SM gets
        // ceil(tiles * n / sms)) times the planes each streams; otherwise the
        // occ resident CTAs of an SM run side by side, and the time goes with
        // the waves of sms * occ CTAs
        int64_t per_slot = (tiles * n + slots - 1) / slots;
        double len = (double)nout / n + 2.0 * r * depth + depth;
        double cost = (double)per_slot * len;
        if (n == 1 || cost < best_cost * 0.98) { best = n; best_cost = cost; }
    }
    return best;
}

// longest unit of the round split (planes; measured on GB300: units of 1024
// planes ran 1-5% slower than the grid split at fused depths 1-3, units of
// 341 planes 5% faster at depth 4)
constexpr double kMaxUnit = 384;

void choose_work_split(LaunchShape& ls, int64_t nout, int r, int depth, int sms, int occ, int* split) {
    *split = 0;
    const int64_t tiles = (int64_t)ls.grid.x * ls.grid.y;
    if (tiles <= 0 || nout <= 0 || sms <= 0) return;
    const char* pin = std::getenv("SO2DR_WORK_SPLIT");
    // grid split: segments by the shared-SM model, or by waves of resident
    // CTAs (SO2DR_WORK_SPLIT=waves)
    const bool waves = pin && std::strcmp(pin, "waves") == 0;
    const int nseg = choose_segments(tiles, nout, r, depth, sms, occ, !waves);
    const double ovh = 2.0 * r * depth + depth;
    const double cost_grid = (double)((tiles * nseg + sms - 1) / sms) * ((double)nout / nseg + ovh);
    // round split: G = sms * occ CTAs take the tiles x n units in rounds;
    // each unit of the last, partial round is cut into floor(G / rem) pieces
    const int64_t occ1 = occ > 0 ? occ : 1, G = (int64_t)sms * occ1;
    int best_n = 0;
    double best = 0;
    for (int n = 1; n <= 64 && n <= nout; ++n) {
        const int64_t units = tiles * n, F = units / G, rem = units - F * G;
        const double len = std::ceil((double)nout / n);
        // units of more than kMaxUnit planes let neighbouring CTAs drift
        // apart along axis 0, and the halo rows they share then miss in L2
        if (len > kMaxUnit && n < nout) continue;
        double cost = (double)F * (len + ovh);
        if (rem) cost += std::ceil(len / (double)(G / rem)) + ovh;
        cost *= (double)occ1;
        if (best_n == 0 || cost < best * 0.98) { best_n = n; best = cost; }
    }
    bool rounds = best_n > 0 && best < cost_grid * 0.97;
    if (pin && (std::strcmp(pin, "grid") == 0 || waves)) rounds = false;
    if (pin && std::strcmp(pin, "rounds") == 0) rounds = true;
    if (rounds) {
        ls.grid = dim3((unsigned)G, 1, 1);
        *split = best_n;
    } else {
        ls.grid.z = (unsigned)nseg;
    }
    // radius 2 at one level: registers for two CTAs per SM, not three, where
    // the launch has no more (star3d_tb.cuh)
    ls.small = r == 2 && depth == 1 && !ls.ragged && (int64_t)ls.grid.x * ls.grid.y * ls.grid.z <= 2 * (int64_t)sms;
}

// FP64 launches of up to this many cells get a tile of their own.  Us a launch,
// the grid's tile / this one / generic kernel: variable coefficients, two levels
// 38x39x32 57.9 / 25.2 / 40.9, 4x256x256 60 / 35 / 39, 20x256x256 142 / 121 /
// 135, four levels 8x256x256 165 / 115 / 147; radius 1 48^3 one level 20.9 /
// 12.3 / 18.9, radius 2 48^3 31.3 / 15.4 / 25.3, 10x512x512 94 / 64 / 88.
// Larger ones keep the grid's tile (64x512x512 radius 4 1106 / 1181 / 1450), and
// so does FP32, whose rows cost little beside a phase (variable coefficients
// 64^3 one level 12.5 / 16.4 / 27.2).
constexpr double kPlaneFitCells = 3e6;

void plane_fit(LaunchShape& ls, int64_t nout, int r, int depth, int64_t ny, int64_t nx, int csize, int sms) {
    if (csize != 8 || sms <= 0 || nout <= 0 || (double)nout * (double)ny * (double)nx > kPlaneFitCells) return;
    plane_shape(ls, r, depth, ny, nx, csize, nout, sms);
}

// Launches of up to this many cells may take the 2-row tile (radius 1 fused,
// radius 3 at one level).  In-core Gcell-steps/s, 4 rows / 2 rows: four levels
// 48x80x132 89 / 96, 64^3 50 / 56, 96^3 153 / 155, 128^3 252 / 186, 160^3 two
// levels 329 / 298; radius 3 64^3 18.3 / 21.3, 128^3 111 / 99.
constexpr double kSmallCells = 1e6;

bool star_small(LaunchShape& ls, int64_t nout, int64_t ny, int64_t nx, int r, int depth, int esize, int sms) {
    if (sms <= 0 || nout <= 0 || (double)nout * (double)ny * (double)nx > kSmallCells || std::getenv("SO2DR_WORK_SPLIT")) return false;
    LaunchShape t = ls;
    switch (r * 16 + depth) {
        case 18: fast_shape<1, 2, true>(t, ny, nx, esize); break;
        case 19: fast_shape<1, 3, true>(t, ny, nx, esize); break;
        case 20: fast_shape<1, 4, true>(t, ny, nx, esize); break;
        case 49: fast_shape<3, 1, true>(t, ny, nx, esize); break;
        default: return false;
    }
    if (!t.ok) return false;
    // A CTA's time goes with the planes it streams (segment, halo, pipeline
    // fill); a second CTA on the same SM costs it about 60% more.
    const double ovh = 2.0 * r * depth + depth;
    const int64_t tiles = (int64_t)t.grid.x * t.grid.y;
    double best = 0;
    int best_n = 0;
    for (int n = 1; n <= 64 && n <= nout; ++n) {
        const int64_t c = (tiles * n + sms - 1) / sms;
        const double cost = ((double)((nout + n - 1) / n) + ovh) * (3.6 * (double)(c / 2) + 2.2 * (double)(c % 2));
        if (!best_n || cost < best * 0.98) { best_n = n; best = cost; }
    }
    // Its planes are quicker (a 4-row CTA's plane takes 1.29 times as long at
    // three and four levels, 1.4 times at the others), but it cuts a plane into
    // more tiles and so the planes into fewer, longer segments; and on a long
    // segment the 4-row kernel's straight-line phases win.  Us a launch, 4 rows
    // / 2 rows: three levels 120x129x16 16.4 / 18.5, 24x512x24 15.0 / 16.4,
    // 64^3 16.2 / 14.5, 600x40x24 22.5 / 24.6; four levels 185x154x16 30.7 /
    // 36.9, 300x48x48 23.9 / 24.6; two levels 2000x20x24 22.5 / 28.7, 60x200x32
    // 13.5 / 12.8; radius 3 185x154x16 16.4 / 18.4.  (Ragged rows: the 2-row
    // tile, three levels 140x200x33 34.8 / 32.8.)
    if (!ls.ragged) {
        const int64_t t4 = (int64_t)ls.grid.x * ls.grid.y;
        const int n4 = choose_segments(t4, nout, r, depth, sms, 1, true);
        const double cost4 = (double)((t4 * n4 + sms - 1) / sms) * ((double)((nout + n4 - 1) / n4) + ovh);
        if (best > cost4 * 2.2 * (r == 1 && depth > 2 ? 1.29 : 1.4) || nout > (12 + depth) * (int64_t)best_n) return false;
    }
    t.grid.z = (unsigned)best_n;
    ls = t;
    return true;
}

void choose_row_split(LaunchShape& ls, int64_t nout, int r, int depth, int csize, int sms, int occ, StencilArgs& a) {
    const int64_t strips = ls.grid.x;
    const int64_t slots = (int64_t)kRowWarps * (occ > 0 ? occ : 1), G = slots * (sms > 0 ? sms : 1);
    // rows a segment streams beyond its own, in units of a row at full depth:
    // the halo (computed by half of the levels on average), the staging fill
    // and the start of a CTA
    const double ovh = 1.0 * r * depth + 8;
    a.split = 1;
    a.split2 = 0;
    a.split_at = nout;
    // Enough rows: one round of long segments over 65% of the rows, one per
    // resident warp, then short ones (a quarter of that length)
    const int64_t m = (strips + G - 1) / G;
    const int64_t n1 = m * G / strips > 0 ? m * G / strips : 1, at = nout * 65 / 100;
    const double len1 = (double)at / (double)n1;
    if (len1 >= 3.0 * ovh) {
        const double len2 = len1 / 4 > 1.5 * ovh ? len1 / 4 : 1.5 * ovh;
        a.split = (int)n1;
        a.split_at = at;
        a.split2 = (int)((double)(nout - at) / len2 + 1);
    } else {
        // Few rows: equal segments.  From wmin units on the warps of an SM
        // share its arithmetic rate, below it each runs at its own pace.
        const int64_t wmin = csize == 8 ? 4 : (slots < 12 ? slots : 12);
        double best = -1;
        for (int64_t q = 1; q <= 4 * slots; q += q < slots ? 1 : slots) {
            int64_t n = q * (sms > 0 ? sms : 1) / strips;
            if (n < 1) n = 1;
            if (n > nout) n = nout;
            const int64_t per_sm = (strips * n * slots + G - 1) / G;
            int64_t busy = per_sm <= slots ? (per_sm > wmin ? per_sm : wmin) : (per_sm + slots - 1) / slots * slots;
            double uneven = 1.0;
            if (csize == 8 && per_sm <= slots) {
                // FP64: a CTA's warps fill an SM, so whole CTAs per SM count; and
                // with fewer than the SMs hold evenly, some get one more all the
                // same (134 to 138 CTAs took 1.4 times as long a row as 144 to 149).
                // Us a launch with fewer / even CTAs: 9-point box, four levels,
                // 600x12800 847 / 572, radius 1 star 484 / 321
                const int64_t ctas = (strips * n + kRowWarps - 1) / kRowWarps, lev = (ctas + sms - 1) / sms;
                busy = kRowWarps * lev;
                if (ctas < 0.93 * lev * sms) uneven = 1.0 + 0.4 / lev;
            }
            const double cost = (double)busy * ((double)((nout + n - 1) / n) + ovh) * uneven;
            if (best < 0 || cost < best * 0.98) { a.split = (int)n; best = cost; }
        }
    }
    ls.grid.x = (unsigned)((strips * (a.split + a.split2) + kRowWarps - 1) / kRowWarps);
}

bool tile2d_short(LaunchShape& ls, int shape, int64_t nout, int64_t nx, int r, int depth, int csize, int sms) {
    // Rows of 32 columns per SM up to which the tile is the faster one
    // (in-core Gcell-steps/s, strips / tile).  FP64, fused: 80x512 radius 1, 4
    // levels 5.6 / 15.7, 512^2 28 / 43, 1024^2 60 / 73 (215 rows per SM).
    // FP64, one level: the tile at any size (us a launch, strips / tile /
    // generic kernel: radius 1 star 4096^2 210 / 174 / 490, 9-point box 300x12800
    // 127 / 76 / 111, radius 4 star 75x3882 43 / 21 / 35, 8000x8192 2580 / 2130 /
    // 2659, 81-point box 4096^2 3681 / 2758 / 3200), but the 25-point box up to
    // 1024 rows (300x12800 357 / 226 / 281; 2001x5003 579 / 612 / 646).  FP64, two
    // levels of radius 3 and 4: 81-point box 500x6000 (618 rows) 1255 / 1155 /
    // 1233, 2000^2 1578 / 1623 / 1798; 49-point box 1000x3882 (802 rows) 872 /
    // 946 / 1072; ragged rows 81-point box 2001x5003 (2067 rows) 4613 / 3959 /
    // 4104, radius 3 star 763 / 601 / 1209.  FP32: 81-point box,
    // one level 512^2 14.0 / 18.8, 1024^2 49 / 52; radius 3, 4 levels,
    // 701x1003 93 / 106; 9-point box, 8 levels 512^2 74 / 85 (54 rows), 1024^2
    // 272 / 219; radius 1, 4 levels 80x512 18 / 20, 256^2 (13 rows) 26 / 25,
    // 512^2 94 / 72.
    const int H = r * depth;
    const int64_t limit = csize == 8 ? (depth == 1 ? (shape == kBox2D && r == 2 ? 1024 : 1 << 30) : r > 2 ? (ls.ragged ? 2200 : 640) : 256)
                          : (shape == kBox2D && r >= 3) || H >= 12 ? 160
                          : H >= 6 ? 60 : depth > 1 ? 12 : 0;
    const int64_t gx = (nx + kTileX - 1) / kTileX;
    if (sms <= 0 || nout <= 0 || gx * nout > limit * sms) return false;
    double best = 0;
    int best_ty = 0;
    for (int ty = 4; ty <= 64; ++ty) {
        if (tile2d_smem(r, depth, ty, csize) > kSmemLimit) break;
        const int64_t gy = (nout + ty - 1) / ty;
        if (gy > 65535) continue;
        double work = 0;
        for (int l = 1; l <= depth; ++l) work += (double)(kTileX + 2 * (H - l * r)) * (ty + 2 * (H - l * r));
        const double cost = (double)((gx * gy + sms - 1) / sms) * (work + 256.0);
        if (!best_ty || cost < best) { best_ty = ty; best = cost; }
    }
    if (!best_ty) return false;
    ls.lx = kTileX + 2 * H;
    ls.ly = best_ty + 2 * H;
    ls.tx = kTileX;
    ls.ty = best_ty;
    ls.block = dim3(kTileThreads, 1, 1);
    ls.smem = (size_t)tile2d_smem(r, depth, best_ty, csize);
    ls.grid = dim3((unsigned)gx, (unsigned)((nout + best_ty - 1) / best_ty), 1);
    ls.fast = kFastTile2D;
    return true;
}

cudaError_t launch_stencil(int dtype, int shape, int r, const StencilArgs& a, const LaunchShape& ls,
                           cudaStream_t s) {
    if (ls.fast == kFastStar3D) switch (dtype) {
        case SO2DR_F32: return ls.ragged ? launch_star3d_ragged_f32(r, a, ls, s) : launch_star3d_f32(r, a, ls, s);
        case SO2DR_BF16: return ls.ragged ? launch_star3d_ragged_bf16(r, a, ls, s) : launch_star3d_bf16(r, a, ls, s);
        case SO2DR_F16: return ls.ragged ? launch_star3d_ragged_f16(r, a, ls, s) : launch_star3d_f16(r, a, ls, s);
        default: return cudaErrorInvalidValue;
    }
    if (ls.fast == kFastRow2D || ls.fast == kFastTile2D) switch (dtype) {
        case SO2DR_F64: return launch_row2d_f64(shape, r, a, ls, s);
        case SO2DR_F32: return launch_row2d_f32(shape, r, a, ls, s);
        case SO2DR_BF16: return launch_row2d_bf16(shape, r, a, ls, s);
        case SO2DR_F16: return launch_row2d_f16(shape, r, a, ls, s);
        default: return cudaErrorInvalidValue;
    }
    switch (dtype) {
        case SO2DR_F64: return launch_stencil_f64(shape, r, a, ls, s);
        case SO2DR_F32: return launch_stencil_f32(shape, r, a, ls, s);
        case SO2DR_BF16: return launch_stencil_bf16(shape, r, a, ls, s);
        case SO2DR_F16: return launch_stencil_f16(shape, r, a, ls, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace so2dr
