// plane_tb.cuh -- plane-streaming temporal-blocking kernel for the 3D stencils
// the register-streaming star kernel does not cover: FP64 stars and the
// variable-coefficient star (FP32 and FP64), any row length.
//
// The on-chip temporal blocking of Sec. III / Sec. IV-A with the levels'
// windows in shared memory:
//  * a CTA of 16 warps owns a loaded tile of LX x ly cells (the halo of
//    R*depth cells each side included) and streams the planes of axis 0.  A
//    thread's cells share one column and lie 512/LX rows apart, so that every
//    index is a 32-bit offset from per-thread constants;
//  * every level keeps 2R+2 planes: the 2R+1 the level above reads and the one
//    being written.  Level l works R+1 planes behind level l-1, on planes
//    completed in earlier phases, so one barrier per plane serves all levels;
//  * the next input plane travels in registers during the phase and is stored
//    at the start of the next one, which hides its latency;
//  * a level computes only the rows its successors need (the compute-area
//    adjustment of Algorithm 1): rows outside are skipped by whole warps.
// FP64 stars are bound by the FP64 units (measured 1.7 lanes per clock and SM:
// 0.52 T FMA/s), so the tile is chosen for the least recomputed halo; the
// variable-coefficient star is bound by its six coefficient loads per cell and
// level, which mostly hit L2.  Gcell-steps/s in core, generic kernel / this
// one: FP64 radius 2, two levels, 150x131x157 11.7 / 20.9; FP64 256^3, radius 1
// one level 47.9 / 54.3, four levels 36.8 / 38.9, radius 4 11.2 / 14.9;
// variable coefficients 243x251x262, four levels 65.5 / 131 (FP32), one level
// 54.4 / 92.8, FP64 two levels 22.3 / 25.7.
// Per-cell arithmetic order: the generic kernel's (stencil.cuh).
#pragma once

#include "stencil.cuh"

namespace so2dr {

constexpr int kPlaneThreads = 512;
constexpr int kPlaneMaxRows = 8;  // rows per thread

// Shared-memory bytes of a launch.
inline int64_t plane_smem_bytes(int r, int depth, int lx, int ly, int csize) {
    return (int64_t)depth * (2 * r + 2) * lx * ly * csize;
}

template <typename T, int R, int SHAPE, int LX>
__global__ void __launch_bounds__(kPlaneThreads, 1) plane_tb_kernel(const StencilArgs a) {
    using C = typename Compute<T>::type;
    constexpr int NS = 2 * R + 2;             // planes per level window
    constexpr int RS = kPlaneThreads / LX;    // row step of a thread's cells
    extern __shared__ __align__(16) unsigned char smem_plane[];
    C* win = reinterpret_cast<C*>(smem_plane);  // [depth][NS][ly][LX]

    const int ly = a.ly, depth = a.depth, tile = LX * ly, H = R * depth;
    const int nx = (int)a.nx, ny = (int)a.ny, n0 = (int)a.n0;
    const int64_t plane = a.ny * a.nx;
    const int lx_ = threadIdx.x % LX, row0 = threadIdx.x / LX;
    const int gx = (int)blockIdx.x * a.tx - H + lx_, gy0 = (int)blockIdx.y * a.ty - H;
    const bool xin = gx >= 0 && gx < nx, xint = gx >= R && gx < nx - R;
    const T* in = static_cast<const T*>(a.in);
    T* out = static_cast<T*>(a.out);
    const C* coef = static_cast<const C*>(a.coef);

    // axis-0 segment of this CTA: outputs [zs, ze), streamed over [za, zb)
    const int in_lo = (int)a.in_lo, in_hi = (int)a.in_hi;
    const int64_t nout = a.out_hi - a.out_lo;
    const int zs = (int)(a.out_lo + nout * blockIdx.z / gridDim.z);
    const int ze = (int)(a.out_lo + nout * (blockIdx.z + 1) / gridDim.z);
    const int za = zs - H > in_lo ? zs - H : in_lo;
    const int zb = ze + H < in_hi ? ze + H : in_hi;
    int64_t slot = (a.in_slot0 + (za - in_lo)) % a.in_cap;  // of the next plane to load
    // slot of the coefficient plane za - R (level 1 in phase 0; phases before
    // plane za never use it)
    const int ccap = SHAPE == kVarcoef3D ? (int)a.coef_cap : 1;
    int cslot = 0;
    if (SHAPE == kVarcoef3D) {
        int64_t c0 = (a.coef_slot0 + (za - R - a.coef_lo)) % a.coef_cap;
        cslot = (int)(c0 < 0 ? c0 + a.coef_cap : c0);
    }

    C pre[kPlaneMaxRows];
    auto load = [&](int z) {  // my cells of plane z into registers, zeros outside the grid
        const T* src = in + slot * plane;
#pragma unroll
        for (int i = 0; i < kPlaneMaxRows; ++i) {
            const int r = row0 + i * RS, gy = gy0 + r;
            pre[i] = C(0);
            if (r < ly && z < zb && xin && gy >= 0 && gy < ny) pre[i] = load_as<T, C>(src + (int64_t)gy * nx + gx);
        }
        if (++slot == a.in_cap) slot = 0;
    };
    auto put = [&](int b) {  // ... and from there into slot b of the input window
#pragma unroll
        for (int i = 0; i < kPlaneMaxRows; ++i) {
            const int r = row0 + i * RS;
            if (r < ly) win[b * tile + r * LX + lx_] = pre[i];
        }
    };
    load(za);
    put(0);
    load(za + 1);
    __syncthreads();

    // level l handles plane za + p - R - (l-1)(R+1) in phase p; the last one
    // ends with plane ze - 1
    const int nph = ze - za + R + (depth - 1) * (R + 1);
    for (int p = 0; p < nph; ++p) {
        // slot of plane za + q: q mod NS; the one of plane za + p + 1 held a
        // plane last read in phase p - 1
        put((p + 1) % NS);
        load(za + p + 2);
        for (int l = 1; l <= depth; ++l) {
            const int q = p - R - (l - 1) * (R + 1), z = za + q;
            const int lo = za > in_lo ? za + l * R : (a.edge_lo ? 0 : in_lo + l * R);
            const int hi = zb < in_hi ? zb - l * R : (a.edge_hi ? n0 : in_hi - l * R);
            if (z < lo || z >= hi) continue;
            const bool last = l == depth;
            if (last && (z < zs || z >= ze)) continue;
            const C* wl = win + (l - 1) * NS * tile;
            const int b = q % NS;  // (q >= 0: z >= lo >= za)
            const C* wp[2 * R + 1];
#pragma unroll
            for (int d = -R; d <= R; ++d) {
                int s = b + d;
                s += s < 0 ? NS : 0;
                s -= s >= NS ? NS : 0;
                wp[d + R] = wl + s * tile;
            }
            C* wo = win + (l * NS + b) * tile;
            const bool zint = z >= R && z < n0 - R;
            const int m = l * R;
            const bool xl = xin && lx_ >= m && lx_ < LX - m;
            const bool xo = lx_ >= H && lx_ < LX - H;
            T* op = out + (z - a.out_lo) * plane + gx;
            // my rows of the level: r = row0 + i * RS in [m, ly - m) and the
            // grid (the same for a whole warp)
            const int rlo = m > -gy0 ? m : -gy0, rhi = ly - m < ny - gy0 ? ly - m : ny - gy0;
            const int ia = rlo > row0 ? (rlo - row0 + RS - 1) / RS : 0, ib = rhi > row0 ? (rhi - row0 + RS - 1) / RS : 0;
            if constexpr (SHAPE == kVarcoef3D) {
                // the coefficients of three rows are loaded at a time, without
                // a branch (cells off the interior read a clamped address), so
                // that 18 loads a thread are in flight (four levels, FP32: 85
                // Gcell-steps/s with a row's six behind its own branch, 131 so)
                int cs = cslot - (l - 1) * (R + 1);
                while (cs < 0) cs += ccap;
                const C* cp = coef + (int64_t)cs * plane;
                const int cx = gx < 1 ? 1 : gx > nx - 2 ? nx - 2 : gx;
                for (int i0 = ia; i0 < ib; i0 += 3) {
                    C cf[3][6];
#pragma unroll
                    for (int u = 0; u < 3; ++u) {
                        int cy = gy0 + row0 + (i0 + u) * RS;
                        cy = cy < 1 ? 1 : cy > ny - 2 ? ny - 2 : cy;
                        const unsigned off = zint && nx > 2 && ny > 2 ? (unsigned)(cy * nx + cx) : 0u;
#pragma unroll
                        for (int f = 0; f < 6; ++f) cf[u][f] = __ldg(cp + f * a.coef_field_stride + off);
                    }
#pragma unroll
                    for (int u = 0; u < 3; ++u) {
                        if (i0 + u >= ib) break;
                        const int r = row0 + (i0 + u) * RS, gy = gy0 + r, o = r * LX + lx_;
                        if (!xl) continue;
                        // faces (-e0,+e0,-e1,+e1,-e2,+e2), centre 1 - sum
                        const C u0 = wp[R][o];
                        C csum = cf[u][0] + cf[u][1];
                        csum = csum + cf[u][2];
                        csum = csum + cf[u][3];
                        csum = csum + cf[u][4];
                        csum = csum + cf[u][5];
                        C v = ((C)1 - csum) * u0;
                        v = fma_c(cf[u][0], wp[0][o], v);
                        v = fma_c(cf[u][1], wp[2 * R][o], v);
                        v = fma_c(cf[u][2], wp[R][o - LX], v);
                        v = fma_c(cf[u][3], wp[R][o + LX], v);
                        v = fma_c(cf[u][4], wp[R][o - 1], v);
                        v = fma_c(cf[u][5], wp[R][o + 1], v);
                        if (!(zint && xint && gy >= R && gy < ny - R)) v = u0;
                        if (!last) wo[o] = v;
                        else if (xo) store_as<T, C>(op + (int64_t)gy * nx, v);
                    }
                }
                continue;
            }
#pragma unroll 2
            for (int i = ia; i < ib; ++i) {
                const int r = row0 + i * RS, gy = gy0 + r, o = r * LX + lx_;
                if (!xl) continue;
                C v;
                if (!(zint && xint && gy >= R && gy < ny - R)) {
                    v = wp[R][o];
                } else {
                    v = (C)a.c[1 + 2 * (R - 1)] * wp[0][o];
#pragma unroll
                    for (int j = R - 1; j >= 1; --j) v = fma_c((C)a.c[1 + 2 * (j - 1)], wp[R - j][o], v);
                    v = fma_c((C)a.c[0], wp[R][o], v);
#pragma unroll
                    for (int j = 1; j <= R; ++j) {
                        v = fma_c((C)a.c[1 + 2 * R + 2 * (j - 1)], wp[R][o - j * LX], v);
                        v = fma_c((C)a.c[2 + 2 * R + 2 * (j - 1)], wp[R][o + j * LX], v);
                    }
#pragma unroll
                    for (int j = 1; j <= R; ++j) {
                        v = fma_c((C)a.c[1 + 4 * R + 2 * (j - 1)], wp[R][o - j], v);
                        v = fma_c((C)a.c[2 + 4 * R + 2 * (j - 1)], wp[R][o + j], v);
                    }
#pragma unroll
                    for (int j = 1; j <= R; ++j) v = fma_c((C)a.c[2 + 2 * (j - 1)], wp[R + j][o], v);
                }
                if (!last) wo[o] = v;
                else if (xo) store_as<T, C>(op + (int64_t)gy * nx, v);
            }
        }
        if (SHAPE == kVarcoef3D && ++cslot == ccap) cslot = 0;
        __syncthreads();
    }
}

}  // namespace so2dr
