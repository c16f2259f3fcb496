// tile2d_tb.cuh -- temporal-blocking kernel for short 2D launches (box and
// star, any type and row length): the whole tile in shared memory.
//
// The streaming kernel (row2d_tb.cuh) pays 2*R*depth halo rows per segment.
// A launch of few rows, cut into enough segments to occupy the SMs, then
// computes several times its useful work, which FP64 (1.7 lanes per clock and
// SM) cannot hide.  Here a CTA loads a square-ish tile with its halo once
// (every load in flight at the same time), runs the fused levels between two
// shared-memory copies with a barrier each, and stores the tile: the halo is
// paid on a tile's rim instead of on every segment's rows.
// Bound by latency: a launch is one load, `depth` barriers and one store.
// Per-cell order: the generic kernel's (stencil.cuh).
#pragma once

#include "stencil.cuh"

namespace so2dr {

constexpr int kTileThreads = 256;
constexpr int kTileX = 32;  // output columns of a tile

// shared-memory bytes of a tile of ty output rows
__host__ __device__ constexpr int tile2d_smem(int r, int depth, int ty, int csize) {
    return 2 * (kTileX + 2 * r * depth) * (ty + 2 * r * depth) * csize;
}

template <typename T, int R, int SHAPE>
__global__ void __launch_bounds__(kTileThreads) tile2d_tb_kernel(const StencilArgs a) {
    using C = typename Compute<T>::type;
    constexpr int W = 2 * R + 1;
    extern __shared__ __align__(16) unsigned char smem_tile[];
    const int H = R * a.depth, lx = kTileX + 2 * H, ly = a.ty + 2 * H, cells = lx * ly;
    C* cur = reinterpret_cast<C*>(smem_tile);
    C* nxt = cur + cells;
    const int nx = (int)a.nx, n0 = (int)a.n0, tid = threadIdx.x;
    const int gx0 = (int)blockIdx.x * kTileX - H;
    const int z0 = (int)a.out_lo + (int)blockIdx.y * a.ty - H;  // grid row of tile row 0
    const int zhi = (int)a.out_hi;
    const T* in = static_cast<const T*>(a.in);
    T* out = static_cast<T*>(a.out);
    auto coef = [&](int k) -> C {
        if constexpr (sizeof(C) == 8) return a.c[k];
        else return a.cf[k];
    };
    // the tile with its halo; zeros outside the grid and the launch's input
    for (int i = tid; i < cells; i += kTileThreads) {
        const int r = i / lx, c = i - r * lx, z = z0 + r, gx = gx0 + c;
        C v = C(0);
        if (z >= a.in_lo && z < a.in_hi && gx >= 0 && gx < nx)
            v = load_as<T, C>(in + ((a.in_slot0 + (z - a.in_lo)) % a.in_cap) * a.nx + gx);
        cur[i] = v;
    }
    __syncthreads();
    for (int l = 1; l <= a.depth; ++l) {
        // rows and columns [m, edge - m) of the tile; a level's cells outside
        // the grid are never read by cells inside (the ring keeps its value)
        const int m = l * R, w = lx - 2 * m, n = w * (ly - 2 * m);
        const bool last = l == a.depth;
        for (int i = tid; i < n; i += kTileThreads) {
            const int r = i / w + m, c = i - (r - m) * w + m, z = z0 + r, gx = gx0 + c;
            const C* p = cur + r * lx + c;
            C v = *p;
            if (z >= R && z < n0 - R && gx >= R && gx < nx - R) {
                if (SHAPE == kStar2D) {
                    v = coef(0) * v;
#pragma unroll
                    for (int j = 1; j <= R; ++j) {
                        v = fma_c(coef(2 * j - 1), p[-j * lx], v);
                        v = fma_c(coef(2 * j), p[j * lx], v);
                    }
#pragma unroll
                    for (int j = 1; j <= R; ++j) {
                        v = fma_c(coef(2 * R + 2 * j - 1), p[-j], v);
                        v = fma_c(coef(2 * R + 2 * j), p[j], v);
                    }
                } else {
                    v = coef(0) * p[-R * lx - R];
#pragma unroll
                    for (int k = 1; k < W * W; ++k) v = fma_c(coef(k), p[(k / W - R) * lx + k % W - R], v);
                }
            }
            if (!last) nxt[r * lx + c] = v;
            else if (z < zhi && gx < nx) store_as<T, C>(out + (z - a.out_lo) * a.nx + gx, v);
        }
        if (last) break;
        __syncthreads();
        C* t = cur;
        cur = nxt;
        nxt = t;
    }
}

}  // namespace so2dr
