// row2d_tb.cuh -- register-streaming temporal-blocking kernel for 2D stencils
// (box and star, radius R, K fused steps per launch), any row length, FP32
// arithmetic on FP32 / BF16 / FP16 storage and FP64 arithmetic on FP64.
//
// The on-chip temporal blocking of Sec. III / Sec. IV-A for the paper's box2d
// workloads (Table III) and the 2D stars, laid out for sm_103a:
//  * a warp owns a strip of 32 lanes x VX columns, of which all but a halo of
//    HXA columns each side are stored, and one axis-0 segment of rows; it
//    streams the rows through its registers.  Column neighbours come from
//    warp shuffles (2R per row and level) and the strips overlap by the halo,
//    so warps never wait on one another: no barrier, and no level touches
//    shared memory.  The launch is a list of strips x segments units, four
//    warps per CTA;
//  * input rows are staged PD rows ahead with cp.async in a ring private to
//    the warp, as 4-element vectors, or element by element where rows are no
//    whole vectors;
//  * box: every level keeps 2R partial sums per cell.  Arriving row y' adds
//    one coefficient row into each of its targets y'-R..y'+R; target y'-R is
//    complete.  The FMAs are scalar, their coefficient a constant-bank
//    operand.  Packed FP32x2 FMAs want it as a register pair: 81 pairs do not
//    fit, and rebuilding them held the 81-point box at 70 of 128 FMAs per
//    clock and SM; at radius 1 and 2, where they fit, they were still slower
//    (9 points, 8 levels: 1548 against 1763 Gcell-steps/s).  The row loop is not unrolled (2R phases of such a body
//    leave the instruction cache: 303 -> 217 Gcell-steps/s at radius 4);
//  * star: the fixed summation order starts at the centre, so a level keeps
//    its last 2R+1 rows and gathers; the row loop is unrolled 2R+1 times and
//    the ring never moves;
//  * a level consumes what the level below completed in the same phase; the
//    independent sums of a level and the other warps of the SM cover the
//    latencies;
//  * cells of the fixed boundary (R columns each side, R rows each end) have
//    their input value at every level: a level that completes such cells takes
//    them from the staged input row, which the ring keeps for R*K rows.
//
// Per-cell order (the generic kernel's, stencil.cuh): box, row by row from
// (-R, -R), the first a multiply; star, centre, (-j, +j) along axis 0 for
// j = 1..R, then (-j, +j) along axis 1.  Every launch, strip and chunk rounds
// identically.
#pragma once

#include "stencil.cuh"
#include "tb_common.cuh"

namespace so2dr {

enum RowKind : int { kRowBox = 0, kRowStar = 1 };

// columns per lane
__host__ __device__ constexpr int row_vx(int kind, int csize, int r, int k) { return kind == kRowBox && csize == 4 && (r == 1 || k == 1) ? 8 : 4; }
// halo columns per side, whole vectors
__host__ __device__ constexpr int row_hxa(int r, int k) { return (r * k + 3) / 4 * 4; }
// rows staged ahead: at one level an SM needs about 44 KB in flight to cover
// the DRAM latency; deeper launches stay longer on each row
__host__ __device__ constexpr int row_pd(int kind, int csize, int r, int k) { return k > 1 ? 4 : row_vx(kind, csize, r, k) == 8 ? 5 : 8; }
// staged rows: the ones ahead, the current one and the R*K a boundary cell
// may be taken back from
__host__ __device__ constexpr int row_nbuf(int kind, int csize, int r, int k) { return row_pd(kind, csize, r, k) + 1 + r * k; }
constexpr int kRowWarps = 4;  // units per CTA

__host__ __device__ constexpr int row_smem(int kind, int csize, int esize, int r, int k) {
    return kRowWarps * 32 * row_vx(kind, csize, r, k) * (row_nbuf(kind, csize, r, k) * esize + csize);
}

template <int KIND, int R, int K, int CS> struct RowShape {
    static constexpr int VX = row_vx(KIND, CS, R, K);
    static constexpr int WX = 32 * VX;          // strip columns
    static constexpr int NT = 32 * kRowWarps;
    static constexpr int HXA = row_hxa(R, K);
    static constexpr int TX = WX - 2 * HXA;     // stored columns per strip
    static constexpr int PD = row_pd(KIND, CS, R, K);
    static constexpr int NBUF = row_nbuf(KIND, CS, R, K);
    // words of per-cell state in registers, and from them the CTAs per SM the
    // compiler is held to (16, 12 or 8 warps; FP64, two lanes per clock and
    // SM, is full with 8)
    static constexpr int STATE = K * (KIND == kRowBox ? 2 * R : 2 * R + 1) * VX * (CS / 4);
    static constexpr int MINB = CS == 8 || STATE >= 84 || (KIND == kRowBox && K > 1 && R > 2 && R * K >= 8) ? 2
                                : STATE >= 60 || (KIND == kRowBox && K > 1 && STATE >= 48) ? 3 : 4;
    static constexpr int UNR = KIND == kRowStar ? 2 * R + 1 : 1;  // phases per turn of the row loop
};

template <typename T, int KIND, int R, int K, bool RAG>
struct Row2D {
    using C = typename Compute<T>::type;
    using S = RowShape<KIND, R, K, (int)sizeof(C)>;
    static constexpr int VX = S::VX, WX = S::WX, PD = S::PD, NBUF = S::NBUF, W = 2 * R + 1, ES = (int)sizeof(T);
    static constexpr int NST = KIND == kRowBox ? 2 * R : W;  // state rows per level
    // 16-bit elements of ragged rows are below cp.async's 4 bytes: they go
    // through registers, one row ahead
    static constexpr bool REGSTAGE = RAG && ES == 2;

    const StencilArgs& a;
    T* sin;   // [NBUF][WX] staged rows of this warp (the row of phase p in slot p % NBUF)
    C* sout;  // [WX] output row on its way to coalesced stores
    int lane, n0, nx, x0, za, zb, slot_next, in_cap, wslot;
    int p_emit, p_lo, p_hi;  // first phase that stores; phases [p_lo, p_hi) complete no boundary cell
    int64_t wrap;            // elements of the circular input buffer
    unsigned ok;             // bit i: my chunk i is inside the grid
    unsigned inx;  // bit e: my column e is an interior column
    bool colb;     // some lane holds a boundary (or outside) column
    const T* in;   // the next row to stage
    T* out;        // the next row to store
    C A[K][NST][VX];  // box: partial sums; star: the last 2R+1 rows
    T rq[VX];         // REGSTAGE: my elements of the next row

    __device__ __forceinline__ explicit Row2D(const StencilArgs& args) : a(args) {}

    // Staged elements of a lane: chunk i of a row starts at strip column
    // col(i); my pointer `in` stands at my chunk 0 of the next row to stage
    // (lanes outside the grid: at its first element, copying nothing).
    static constexpr int VE = RAG ? 1 : ES == 8 ? 2 : 4;  // elements per copy
    static constexpr int NCH = VX / VE;                   // copies per row
    __device__ __forceinline__ int col(int i) const { return VE * (lane + 32 * i); }
    __device__ __forceinline__ bool inside(int i) const { return x0 + col(i) >= 0 && x0 + col(i) < nx; }

    __device__ __forceinline__ void next_row() {
        in += nx;
        if (++slot_next == in_cap) {
            slot_next = 0;
            in -= wrap;
        }
    }

    // REGSTAGE: my elements of row z into rq
    __device__ __forceinline__ void fetch_regs(int z) {
        if (z < zb) {
#pragma unroll
            for (int i = 0; i < NCH; ++i) rq[i] = (ok >> i) & 1u ? in[(x0 + col(i))] : T(0.f);
            next_row();
        }
    }
    __device__ __forceinline__ void put_regs(int b) {
#pragma unroll
        for (int i = 0; i < NCH; ++i) sin[b * WX + col(i)] = rq[i];
    }

    // one commit group per call (empty past the input), so that waiting for
    // all but the newest PD - 1 groups always means: this phase's row landed
    __device__ __forceinline__ void stage(int z, int b) {
        if (z < zb) {
            T* dst = sin + b * WX + col(0);
#pragma unroll
            for (int i = 0; i < NCH; ++i) {
                const bool o = (ok >> i) & 1u;
                const T* src = o ? in + x0 + col(i) : in;
                if constexpr (RAG) cp_async_elem(dst + 32 * VE * i, src, o);
                else if constexpr (ES == 8) cp_async16(dst + 32 * VE * i, src, o);
                else cp_async_vec4(dst + 32 * VE * i, src, o);
            }
            next_row();
        }
        cp_async_commit();
    }

    __device__ __forceinline__ C coef(int k) const {
        if constexpr (sizeof(C) == 8) return a.c[k];
        else return a.cf[k];
    }

    // my cells of the staged row in slot b
    __device__ __forceinline__ void read_row(int b, C (&v)[VX]) const {
        const T* row = sin + b * WX + VX * lane;
#pragma unroll
        for (int i = 0; i < VX; i += 4) {
            if constexpr (ES == 8) {
                const double2 q0 = *reinterpret_cast<const double2*>(row + i), q1 = *reinterpret_cast<const double2*>(row + i + 2);
                v[i] = q0.x; v[i + 1] = q0.y; v[i + 2] = q1.x; v[i + 3] = q1.y;
            } else {
                const float4 q = lds4(row + i);
                v[i] = q.x; v[i + 1] = q.y; v[i + 2] = q.z; v[i + 3] = q.w;
            }
        }
    }

    // values of columns -R .. VX-1+R around my first column
    __device__ __forceinline__ void window(const C (&v)[VX], C (&w)[VX + 2 * R]) const {
#pragma unroll
        for (int e = 0; e < VX; ++e) w[R + e] = v[e];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            w[R - 1 - i] = __shfl_up_sync(0xffffffffu, v[VX - 1 - i], 1);
            w[R + VX + i] = __shfl_down_sync(0xffffffffu, v[i], 1);
        }
    }

    // box, level L: a row arrives with values v; v becomes the row R before
    // it.  Target q (q = 0..2R) is R - q rows before the arrival, which is its
    // coefficient row 2R - q; every sum moves one slot down as its last
    // product is added.
    template <int L>
    __device__ __forceinline__ void arrive_box(C (&v)[VX]) {
        C w[VX + 2 * R], done[VX];
        window(v, w);
#pragma unroll
        for (int q = 0; q < W; ++q) {
            C s[VX];
#pragma unroll
            for (int dx = 0; dx < W; ++dx)
#pragma unroll
                for (int i = 0; i < VX; ++i) {
                    const int k = (2 * R - q) * W + dx;
                    if (q == 2 * R && dx == 0) s[i] = coef(k) * w[i];
                    else s[i] = fma_c(coef(k), w[i + dx], dx == 0 ? A[L][q][i] : s[i]);
                }
#pragma unroll
            for (int i = 0; i < VX; ++i) {
                if (q == 0) done[i] = s[i];
                else A[L][q - 1][i] = s[i];
            }
        }
#pragma unroll
        for (int i = 0; i < VX; ++i) v[i] = done[i];
    }

    // star, level L: a row arrives with values v (ring slot SL); v becomes the
    // row R below it, gathered from the ring
    template <int L, int SL>
    __device__ __forceinline__ void arrive_star(C (&v)[VX]) {
        C w[VX + 2 * R];
#pragma unroll
        for (int i = 0; i < VX; ++i) A[L][SL][i] = v[i];
        constexpr int CT = pmod(SL - R, W);
        window(A[L][CT], w);
#pragma unroll
        for (int i = 0; i < VX; ++i) {
            C s = coef(0) * w[R + i];
#pragma unroll
            for (int j = 1; j <= R; ++j) {
                s = fma_c(coef(2 * j - 1), A[L][pmod(CT - j, W)][i], s);
                s = fma_c(coef(2 * j), A[L][pmod(CT + j, W)][i], s);
            }
#pragma unroll
            for (int j = 1; j <= R; ++j) {
                s = fma_c(coef(2 * R + 2 * j - 1), w[R + i - j], s);
                s = fma_c(coef(2 * R + 2 * j), w[R + i + j], s);
            }
            v[i] = s;
        }
    }

    // levels L..K-1 of the phase in which row y arrives at level 0; v holds
    // what arrives at level L (row y - L*R).  EDGE: the phase may complete
    // boundary cells or lie in the head of the stream, where level L has
    // nothing to do until its arrivals are valid (row za + L*R, or the grid's
    // first row).
    template <int L, int PH, bool EDGE>
    __device__ __forceinline__ void levels(int y, C (&v)[VX]) {
        if constexpr (EDGE)
            if (y - L * R < (za > 0 ? za + L * R : 0)) return;
        if constexpr (KIND == kRowBox) arrive_box<L>(v);
        else arrive_star<L, pmod(PH - L * R, W)>(v);
        if constexpr (EDGE) {
            const int t = y - (L + 1) * R;  // the completed row
            const bool rb = t < R || t >= n0 - R;
            if (colb || rb) {
                C o[VX];
                const int b = wslot - (L + 1) * R;
                read_row(b < 0 ? b + NBUF : b, o);
#pragma unroll
                for (int e = 0; e < VX; ++e)
                    if (rb || !((inx >> e) & 1u)) v[e] = o[e];
            }
        }
        if constexpr (L + 1 < K) levels<L + 1, PH, EDGE>(y, v);
    }

    __device__ __forceinline__ void emit(const C (&v)[VX]) {
        T* ob = out;
        out += nx;
        if constexpr (!RAG && VX == 4) {
            const int j = 4 * lane, gx = x0 + j;
            if (j >= S::HXA && j < S::HXA + S::TX && gx < nx) {
                if constexpr (ES == 8) {
                    reinterpret_cast<double2*>(ob + gx)[0] = make_double2(v[0], v[1]);
                    reinterpret_cast<double2*>(ob + gx)[1] = make_double2(v[2], v[3]);
                } else {
                    st4(ob + gx, make_float4(v[0], v[1], v[2], v[3]));
                }
            }
        } else {
            // through shared memory, so that a warp's stores are contiguous
#pragma unroll
            for (int e = 0; e < VX; ++e) sout[VX * lane + e] = v[e];
            __syncwarp();
            if constexpr (RAG) {
#pragma unroll
                for (int e = 0; e < VX; ++e) {
                    const int j = lane + 32 * e, gx = x0 + j;
                    if (j >= S::HXA && j < S::HXA + S::TX && gx < nx) store_as<T, C>(ob + gx, sout[j]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < VX / 4; ++i) {
                    const int j = 4 * (lane + 32 * i), gx = x0 + j;
                    if (j >= S::HXA && j < S::HXA + S::TX && gx < nx) st4(ob + gx, *reinterpret_cast<const float4*>(sout + j));
                }
            }
        }
    }

    // phase p (PH = p mod UNR): row za + p
    template <int PH>
    __device__ __forceinline__ void phase(int p) {
        const int y = za + p;
        if constexpr (!REGSTAGE) cp_async_wait_group<PD - 1>();
        __syncwarp();  // the other lanes' copies of this row; their reads of the last output row
        C v[VX];
        read_row(wslot, v);
        // the slot of row y + PD held row y - 1 - R*K, last read in phase p - 1
        if constexpr (REGSTAGE) {
            put_regs(wslot + 1 == NBUF ? 0 : wslot + 1);
            fetch_regs(y + 2);
        } else {
            stage(y + PD, wslot + PD >= NBUF ? wslot + PD - NBUF : wslot + PD);
        }
        if (p < p_lo || p >= p_hi) levels<0, PH, true>(y, v);
        else levels<0, PH, false>(y, v);
        if (p >= p_emit) emit(v);
        if (++wslot == NBUF) wslot = 0;
    }
    template <int PH>
    __device__ __forceinline__ void phases(int p, int nph) {
        if (p + PH < nph) phase<PH>(p + PH);
        if constexpr (PH + 1 < S::UNR) phases<PH + 1>(p, nph);
    }

    __device__ __forceinline__ void run(unsigned char* smem) {
        lane = threadIdx.x & 31;
        const int warp = threadIdx.x >> 5;
        nx = (int)a.nx;
        n0 = (int)a.n0;
        sout = reinterpret_cast<C*>(smem) + warp * WX;
        sin = reinterpret_cast<T*>(smem + kRowWarps * WX * sizeof(C)) + warp * NBUF * WX;
        const int strips = (nx + S::TX - 1) / S::TX;
        const int64_t unit = (int64_t)blockIdx.x * kRowWarps + warp;
        if (unit >= (int64_t)strips * (a.split + a.split2)) return;
        const int strip = (int)(unit % strips), seg = (int)(unit / strips);
        x0 = strip * S::TX - S::HXA;
        inx = 0;
#pragma unroll
        for (int e = 0; e < VX; ++e) {
            const int gx = x0 + VX * lane + e;
            if (gx >= R && gx < nx - R) inx |= 1u << e;
        }
        colb = __any_sync(0xffffffffu, inx != (1u << VX) - 1u);
        // axis-0 segment: outputs [zs, ze), streamed over [za, zb).  Sums that
        // a row before za would have reached belong to rows that are never
        // stored: away from the grid's first row the valid rows shrink by R
        // per level, and at it they are boundary rows, taken from the input.
        // The units are a.split long segments over the first a.split_at rows,
        // then a.split2 short ones over the rest: CTAs start in that order, so
        // the short ones even out the SMs' ends.
        const int in_lo = (int)a.in_lo, in_hi = (int)a.in_hi;
        const bool tail = seg >= a.split;
        const int64_t s0 = a.out_lo + (tail ? a.split_at : 0), k = tail ? seg - a.split : seg,
                      len = tail ? a.out_hi - a.out_lo - a.split_at : a.split_at, nk = tail ? a.split2 : a.split;
        const int zs = (int)(s0 + len * k / nk), ze = (int)(s0 + len * (k + 1) / nk);
        if (ze <= zs) return;
        za = zs - K * R > in_lo ? zs - K * R : in_lo;
        zb = ze + K * R < in_hi ? ze + K * R : in_hi;
        in_cap = (int)a.in_cap;
        slot_next = (int)((a.in_slot0 + (za - in_lo)) % a.in_cap);
        wrap = a.in_cap * nx;
        in = static_cast<const T*>(a.in) + (int64_t)slot_next * nx;
        out = static_cast<T*>(a.out) + (zs - a.out_lo) * nx;
        ok = 0;
#pragma unroll
        for (int i = 0; i < NCH; ++i) ok |= inside(i) ? 1u << i : 0u;
        // phase p completes rows za + p - K*R .. za + p - R; rows of the fixed
        // boundary, and the head of the stream, run the EDGE body
        p_emit = zs + K * R - za;
        p_lo = K * R + R - za > 2 * K * R ? K * R + R - za : 2 * K * R;
        p_hi = colb ? 0 : n0 - za;
        wslot = 0;
#pragma unroll
        for (int l = 0; l < K; ++l)
#pragma unroll
            for (int q = 0; q < NST; ++q)
#pragma unroll
                for (int e = 0; e < VX; ++e) A[l][q][e] = C(0);
        if constexpr (REGSTAGE) {
            fetch_regs(za);
            put_regs(0);
            fetch_regs(za + 1);
        } else {
            for (int i = 0; i < PD; ++i) stage(za + i, i);
        }
        const int nph = ze + K * R - za;  // the last output row completes with row ze - 1 + K*R
        for (int p = 0; p < nph; p += S::UNR) phases<0>(p, nph);
        if constexpr (!REGSTAGE) cp_async_wait_all();
    }
};

template <typename T, int KIND, int R, int K, bool RAG>
__global__ void __launch_bounds__(RowShape<KIND, R, K, (int)sizeof(typename Compute<T>::type)>::NT,
                                  RowShape<KIND, R, K, (int)sizeof(typename Compute<T>::type)>::MINB)
    row2d_tb_kernel(const StencilArgs a) {
    extern __shared__ __align__(16) unsigned char smem_row[];
    Row2D<T, KIND, R, K, RAG> k(a);
    k.run(smem_row);
}

}  // namespace so2dr
