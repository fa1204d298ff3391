// Internal declarations shared by the libfftpl translation units.
//
// Layout in device memory (all float32 unless noted, row-major [n][n] maps
// with x fastest):
//   movable cells   w, h                       (m_mov)
//   fixed cells     fix_x, fix_y (m_fix)       macro map M = rho_t F  [n][n]
//   density         D (movable overlap area, float) or Dq (int64, 2^-32 units)
//   spectral        T1 [u/2][y] of (u even, u odd)  (rows transformed along x,
//                   stored transposed), PT, RT [y/2][u] of (y even, y odd)
//                   (columns transformed and inverted)
//                   psi, ex, ey [y][x], rho [y][x] (formed on demand)
//   nets/pins       slabs of nets of equal degree; pin_cell, pin_dx, pin_dy,
//                   pin_slot in slab order (slot base + 32 k + lane);
//                   cell_pin_ptr (m_mov+1), gpin (float2 per pin) for the
//                   deterministic pin-to-cell reduction; gW2 (float2, m_mov)
//                   the atomic one
//   accumulators    acc[ACC_*] doubles, err word
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "fftpl.h"

namespace fftpl {

// ------------------------------------------------------------------ sizes
constexpr int kCellThreads = 256;
// Blocks per SM of the cell kernels (field gather and pin sums): 24 warps of up
// to 80 registers, room for four 32-byte loads in flight per thread and the
// next cell's inputs.  k_cells at 2.2M cells under ncu with 2 / 3 / 4 blocks:
// 48.6 / 39.2 / 45.1 us (4: spills).
constexpr int kCellBlocks = 3;
constexpr int kWaThreads = 256;
// Nets of degree kBigMin..kBigMax take several lanes per net in the WA kernel
// (grp_lanes(d) lanes each, at most 4 pins per lane); the rest one lane.
constexpr int kBigMin = 7;
constexpr int kBigMax = 64;
__host__ __device__ constexpr int grp_lanes(int d) {
    return d <= 8 ? 2 : (d <= 16 ? 4 : (d <= 32 ? 8 : 16));
}

// lanes of a net of degree d in the slab layout
__host__ __device__ constexpr int net_lanes(int d) {
    return d >= kBigMin && d <= kBigMax ? grp_lanes(d) : 1;
}

// accumulator slots (FP64 sums written by the kernels)
enum {
    ACC_N = 0,      // sum B * Psi (times A_b/2 on the host)
    ACC_W,          // WA wirelength
    ACC_HPWL,
    ACC_TAU,        // overflow numerator
    ACC_GN_L1,
    ACC_GW_L1,
    ACC_CHARGE,     // sum (D + M) (times A_b... area units already)
    ACC_DV2,        // ||v_k - v_{k-1}||^2
    ACC_DG2,        // ||g_k - g_{k-1}||^2
    ACC_GINF,       // ||g_k||_inf (as ordered bits of a non-negative double)
    ACC_STEPMAX,    // max |u_{k+1} - v_k|
    ACC_GD,         // g_k . d_k (conjugate-gradient loop)
    ACC_DINF,       // ||d_k||_inf (conjugate-gradient loop)
    ACC_COUNT
};

// the sums an evaluation reports: the first kReportSums quantities
constexpr int kReportSums = ACC_CHARGE + 1;
// where the host mirror holds the number of the report it is from
constexpr int kReportFlag = 31;

// The FP64 sums are striped: a block adds its total to stripe
// (blockIdx & 31), one 128-byte line of kAccStride doubles per stripe, so no
// single address takes every block's atomic; readers add the stripes.
constexpr int kAccStripes = 32;
constexpr int kAccStride = 16;
constexpr int kAccDoubles = kAccStripes * kAccStride;
static_assert(ACC_COUNT <= kAccStride, "accumulator stripe too small");

// device error word bits
enum { ERR_TIMEOUT = 1, ERR_BOUNDS = 2 };

// Bin grid along both axes.  Edges e_k = x0 + k * wb, k <= n, are exact in
// float32 (checked at create), so comparisons against them decide indices
// exactly, and an edge formed as fma(k, wb, x0) or by adding wb to the one
// before it is that same number.
struct Grid {
    int n;
    float x0, y0, wb, hb, inv_wb, inv_hb;
};

__device__ __forceinline__ float edge_at(float lo, float step, int k) {
    return __fadd_rn(lo, __fmul_rn((float)k, step));
}

// Largest k in [-1, n] with e_k <= t (strict: e_k < t), limited to [LO, HI]
// (-1 for NaN, limited alike).  The float estimate q = (t - x0) * (1/w_b) is
// within one of the answer (its relative error is a few 2^-24 and the
// quotient at most n + 1 after the limits), so one comparison against the
// exact edge on each side settles the index.  No branches: a fast path for
// estimates away from an edge, the comparisons otherwise, cost the cell
// kernels more than the comparisons (a warp took both).
template <bool STRICT>
__device__ __forceinline__ int last_edge(float lo, float step, float inv, float kmin, float kmax,
                                         float t) {
    float k = fminf(fmaxf(floorf(__fmul_rn(__fsub_rn(t, lo), inv)), kmin), kmax);
    const float e0 = fmaf(k, step, lo), e1 = fmaf(k + 1.0f, step, lo);
    const bool up = k < kmax && (STRICT ? e1 < t : e1 <= t);
    const bool down = k > kmin && !(STRICT ? e0 < t : e0 <= t);
    return (int)k + (up ? 1 : 0) - (down ? 1 : 0);
}

struct Span {
    float xl, xh, yl, yh;   // float32 cell edges
    int ilo, ihi, jlo, jhi; // clamped bin span (empty if ilo > ihi or jlo > jhi)
};

__device__ __forceinline__ Span cell_span(const Grid& g, float x, float y, float w, float h) {
    Span s;
    float hw = __fmul_rn(0.5f, w), hh = __fmul_rn(0.5f, h);
    s.xl = __fsub_rn(x, hw);
    s.xh = __fadd_rn(x, hw);
    s.yl = __fsub_rn(y, hh);
    s.yh = __fadd_rn(y, hh);
    const float n = (float)g.n;
    s.ilo = last_edge<false>(g.x0, g.wb, g.inv_wb, 0.0f, n, s.xl);
    s.ihi = last_edge<true>(g.x0, g.wb, g.inv_wb, -1.0f, n - 1.0f, s.xh);
    s.jlo = last_edge<false>(g.y0, g.hb, g.inv_hb, 0.0f, n, s.yl);
    s.jhi = last_edge<true>(g.y0, g.hb, g.inv_hb, -1.0f, n - 1.0f, s.yh);
    return s;
}

// Overlap length of [a, b) with bin k (float32 arithmetic, no contraction).
__device__ __forceinline__ float ov_len(float lo, float step, int k, float a, float b) {
    float e0 = edge_at(lo, step, k), e1 = edge_at(lo, step, k + 1);
    float v = __fsub_rn(fminf(b, e1), fmaxf(a, e0));
    return fmaxf(v, 0.0f);
}

// The same overlaps of consecutive bins: with c(e) = e limited to [a, b],
// bin k's is c(e_{k+1}) - c(e_k) (both terms equal, so exactly 0, outside
// the span; inside it the operands of ov_len).
__device__ __forceinline__ float edge_in(float e, float a, float b) {
    return fminf(fmaxf(e, a), b);
}

// x overlaps of the aligned group of four bins 4 q .. 4 q + 3.
__device__ __forceinline__ void quad_ov(const Grid& g, const Span& s, int q, float (&ox)[4]) {
    float e = fmaf((float)(4 * q), g.wb, g.x0), c = edge_in(e, s.xl, s.xh);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        e = __fadd_rn(e, g.wb);
        const float d = edge_in(e, s.xl, s.xh);
        ox[t] = __fsub_rn(d, c);
        c = d;
    }
}

// Four bins of the interleaved field, (E_x, E_y) each: one 32-byte sector (a
// coherent load behind chain_wait, as ld_dep).
struct Field4 {
    float v[8];
};
__device__ __forceinline__ Field4 load_field4(const float2* p) {
    Field4 f;
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(f.v[0]), "=f"(f.v[1]), "=f"(f.v[2]), "=f"(f.v[3]), "=f"(f.v[4]),
                   "=f"(f.v[5]), "=f"(f.v[6]), "=f"(f.v[7])
                 : "l"(p)
                 : "memory");
    return f;
}

__device__ __forceinline__ void field_fma(const float (&ox)[4], float oy, const Field4& f,
                                          float& sx, float& sy) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float o = __fmul_rn(ox[t], oy);
        sx = fmaf(o, f.v[2 * t], sx);
        sy = fmaf(o, f.v[2 * t + 1], sy);
    }
}

// Part of a field gather: groups of four bins q0 .. q1, rows j0 .. j1.
__device__ __forceinline__ void gather_part(const Grid& g, const Span& s, int q0, int q1, int j0,
                                            int j1, const float2* __restrict__ E2, float& sx,
                                            float& sy) {
    for (int q = q0; q <= q1; ++q) {
        float ox[4];
        quad_ov(g, s, q, ox);
        const float2* p = E2 + (size_t)j0 * g.n + 4 * q;
        float e = fmaf((float)j0, g.hb, g.y0), c = edge_in(e, s.yl, s.yh);
        for (int j = j0; j <= j1; ++j, p += g.n) {
            const Field4 f = load_field4(p);
            e = __fadd_rn(e, g.hb);
            const float d = edge_in(e, s.yl, s.yh);
            field_fma(ox, __fsub_rn(d, c), f, sx, sy);
            c = d;
        }
    }
}

// Field gather of one cell: sum_b ov(i,b) E2[b] over its bin span, E2 the
// interleaved (E_x, E_y) map.  A cell's bins lie in lines of their own, so
// every lane of a load costs the L1 one wavefront: whole sectors (aligned
// groups of four bins, zero weights outside the span) take about half as
// many as one load per bin.  What bounds it is the latency of those loads and
// the L1's wavefronts (78 % busy), so the first two groups of the first two
// rows (nearly every cell) go out together.  Against one 8-byte load per bin
// in chunks of 2 x 4 bins, one cell per thread: k_cells at 2.2M cells, n = 2048
// 52.8 -> 39.2 us (39.1M -> 22.2M warp instructions), at 210K cells 9.7 -> 8.8,
// k_gather at 5M cells, n = 4096 (E2 larger than the L2) 119 -> 111 us.
__device__ __forceinline__ float2 gather_span(const Grid& g, const Span& s,
                                              const float2* __restrict__ E2) {
    if (s.jlo > s.jhi || s.ilo > s.ihi) return make_float2(0.0f, 0.0f);
    const int q0 = s.ilo >> 2, q1 = s.ihi >> 2;
    const bool two_q = q0 < q1, two_j = s.jlo < s.jhi;
    const float2* p = E2 + (size_t)s.jlo * g.n + 4 * q0;
    Field4 f00 = load_field4(p), f01 = {}, f10 = {}, f11 = {};
    if (two_q) f01 = load_field4(p + 4);
    if (two_j) f10 = load_field4(p + g.n);
    if (two_q && two_j) f11 = load_field4(p + g.n + 4);
    const float e0 = fmaf((float)s.jlo, g.hb, g.y0), e1 = e0 + g.hb, e2 = e1 + g.hb;
    const float c0 = edge_in(e0, s.yl, s.yh), c1 = edge_in(e1, s.yl, s.yh),
                c2 = edge_in(e2, s.yl, s.yh);
    const float oa = __fsub_rn(c1, c0), ob = __fsub_rn(c2, c1);
    float sx = 0.0f, sy = 0.0f, ox[4];
    quad_ov(g, s, q0, ox);
    field_fma(ox, oa, f00, sx, sy);
    if (two_j) field_fma(ox, ob, f10, sx, sy);
    if (two_q) {
        quad_ov(g, s, q0 + 1, ox);
        field_fma(ox, oa, f01, sx, sy);
        if (two_j) field_fma(ox, ob, f11, sx, sy);
    }
    if (q0 + 2 <= q1) gather_part(g, s, q0 + 2, q1, s.jlo, s.jhi, E2, sx, sy);
    if (s.jlo + 2 <= s.jhi)
        gather_part(g, s, q0, min(q0 + 1, q1), s.jlo + 2, s.jhi, E2, sx, sy);
    return make_float2(sx, sy);
}

// What a cell kernel reads of a cell in the caller's order, loaded one round
// ahead of its use: the cell kernels run a fixed grid, each thread striding
// over the cells.
struct CellIn {
    float x, y, w, h;
    int r;
};
__device__ __forceinline__ CellIn load_cell(int i, int m, const float* __restrict__ x,
                                            const float* __restrict__ y,
                                            const float* __restrict__ w,
                                            const float* __restrict__ h,
                                            const int* __restrict__ rank) {
    CellIn c = {};
    if (i < m) {
        c.x = __ldg(x + i);
        c.y = __ldg(y + i);
        c.w = __ldg(w + i);
        c.h = __ldg(h + i);
        if (rank) c.r = __ldg(rank + i);
    }
    return c;
}

// ------------------------------------------- programmatic dependent launch
// A kernel launched with launch_chain may start while the kernel before it in
// the stream still runs, from the moment every block of that one has called
// chain_trigger; what it reads of it comes after chain_wait, which returns
// when that kernel has completed.  Every kernel of a chain calls both (chain_wait
// first among its reads), so that its completion also means its
// predecessors'.  Both are no-ops in a plain launch.  Only where the kernel
// before is the launch's single dependency: never after a join with another
// stream.
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void chain_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// What the kernel before in a chain writes is read with these: coherent (the
// read-only path, ld.global.nc and __ldg, is for data that no one writes while
// the kernel lives, and a kernel of a chain lives while its predecessor still
// writes) and volatile (no compiler moves them above chain_wait).
__device__ __forceinline__ float ld_dep(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_dep(const float2* p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_dep(const float4* p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ longlong2 ld_dep(const longlong2* p) {
    longlong2 v;
    asm volatile("ld.global.v2.s64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

template <typename... P, typename... A>
cudaError_t launch_chain(void (*kern)(P...), int blocks, int threads, size_t smem, cudaStream_t s,
                         bool chain, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// --------------------------------------------------- double-float sums
// An unevaluated sum hi + lo of two floats (error-free transformations:
// Knuth's TwoSum and Dekker's Fast2Sum).  Used to keep the grid-wide FP64
// reductions accurate without FP64 arithmetic in the inner loops.
struct dfloat {
    float hi, lo;
};

__device__ __forceinline__ dfloat df_zero() { return {0.0f, 0.0f}; }

__device__ __forceinline__ dfloat df_add(dfloat a, float b) {
    float s = __fadd_rn(a.hi, b);
    float bb = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    float lo = __fadd_rn(a.lo, e);
    float hi = __fadd_rn(s, lo);
    return {hi, __fsub_rn(lo, __fsub_rn(hi, s))};
}

__device__ __forceinline__ dfloat df_add(dfloat a, dfloat b) {
    dfloat r = df_add(a, b.hi);
    return df_add(r, b.lo);
}

// The same for the few terms of a loop's one round: the rounding errors are
// added up beside the sum without renormalising (Sum2 of Ogita, Rump and Oishi,
// 2005, as if in twice the precision; 7 operations a term instead of 10).
__device__ __forceinline__ void sum2_add(dfloat& a, float b) {
    const float s = __fadd_rn(a.hi, b);
    const float bb = __fsub_rn(s, a.hi);
    a.lo = __fadd_rn(a.lo, __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
    a.hi = s;
}

__device__ __forceinline__ double* acc_stripe(double* acc, int q) {
    return acc + (blockIdx.x & (kAccStripes - 1)) * kAccStride + q;
}

// Max of non-negative doubles through their ordered bit patterns.
__device__ __forceinline__ void atomic_max_nonneg(double* dst, double v) {
    atomicMax(reinterpret_cast<unsigned long long*>(dst),
              (unsigned long long)__double_as_longlong(v));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the first n lanes (the others hold 0).
__device__ __forceinline__ double warp_sum_f64(double v, int n) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (o < n) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// *p += (a, b) as one relaxed, device-scope 8-byte vector reduction with no
// return value (the same operation as atomicAdd on a float2, which is issued
// as a returning atomic and so holds its destination registers until the
// answer comes back).
__device__ __forceinline__ void red_add_f2(float2* p, float a, float b) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}

// *p += (a, b, c, d), 16 bytes, likewise.
__device__ __forceinline__ void red_add_f4(float* p, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c),
                 "f"(d)
                 : "memory");
}

// *p += v as a relaxed, device-scope reduction with no return value.
__device__ __forceinline__ void red_add_f64(double* p, double v) {
    asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

// Sums of non-negative per-thread values a and b over each warp (a float32
// tree: relative error at most 5 units in the last place for non-negative
// terms, besides what the caller's own sums over a thread's items lost: kernels
// whose threads take a number of items that grows with the instance keep them
// as double-float pairs); lane 0 adds each nonzero warp total in FP64 to the stripe of
// quantity qa / qb (qb < 0: none) chosen by the warp's global index.  No
// block-wide barrier, and the atomics spread over 32 lines.
__device__ __forceinline__ void block_acc2(float a, float b, double* acc, int qa, int qb) {
    a = warp_sum(a);
    b = warp_sum(b);
    if ((threadIdx.x & 31) == 0) {
        unsigned gw = (blockIdx.x * ((blockDim.x + 31) >> 5)) + (threadIdx.x >> 5);
        double* st = acc + (gw & (kAccStripes - 1)) * kAccStride;
        if (qa >= 0 && a != 0.0f) red_add_f64(st + qa, (double)a);
        if (qb >= 0 && b != 0.0f) red_add_f64(st + qb, (double)b);
    }
}

__device__ __forceinline__ void block_acc1(float a, double* acc, int qa) {
    block_acc2(a, 0.0f, acc, qa, -1);
}

// Deterministic (order-free) reduction for the deterministic mode: each
// block sums its threads in a fixed tree and stores its totals in its own
// slot of part[]; the block that draws the last ticket (after a fence) adds
// all slots in index order and stores the totals in stripe 0.  Nothing
// waits.  part == nullptr selects the striped atomics of block_acc2.
struct DetRed {
    double* part;       // [2][cap] block totals
    unsigned* ticket;   // zero between launches (the last block resets it)
    int cap;            // capacity in blocks
};

__device__ __forceinline__ void reduce2(float a, float b, double* acc, int qa, int qb,
                                        const DetRed& dr) {
    if (!dr.part) {
        block_acc2(a, b, acc, qa, qb);
        return;
    }
    // every sum in FP64 is a tree over the lanes of the first warp (one thread
    // adding the warps' totals in turn: wirelength alone at 34K cells 21.0 ->
    // 19.8 us, 2.2M 242 -> 237)
    __shared__ float s_f[2][32];
    __shared__ double s_d[2][32];
    __shared__ bool s_last;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    a = warp_sum(a);
    b = warp_sum(b);
    __syncthreads();
    if (l == 0) {
        s_f[0][w] = a;
        s_f[1][w] = b;
    }
    __syncthreads();
    if (w == 0) {
        const double ta = warp_sum_f64(l < nw ? (double)s_f[0][l] : 0.0, nw);
        const double tb = warp_sum_f64(l < nw ? (double)s_f[1][l] : 0.0, nw);
        if (l == 0) {
            dr.part[blockIdx.x] = ta;
            dr.part[dr.cap + blockIdx.x] = tb;
            __threadfence();
            unsigned t = atomicAdd(dr.ticket, 1u);
            s_last = (t == gridDim.x - 1);
            if (s_last) *dr.ticket = 0u;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double ta = 0.0, tb = 0.0;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) {
        ta += __ldcg(dr.part + k);
        tb += __ldcg(dr.part + dr.cap + k);
    }
    // fixed-order tree over the block (warps, then warp totals)
    ta = warp_sum_f64(ta, 32);
    tb = warp_sum_f64(tb, 32);
    if (l == 0) {
        s_d[0][w] = ta;
        s_d[1][w] = tb;
    }
    __syncthreads();
    if (w != 0) return;
    ta = warp_sum_f64(l < nw ? s_d[0][l] : 0.0, nw);
    tb = warp_sum_f64(l < nw ? s_d[1][l] : 0.0, nw);
    if (l == 0) {
        if (qa >= 0) acc[qa] = ta;
        if (qb >= 0) acc[qb] = tb;
        __threadfence();
    }
}

// a dfloat collapsed to the nearest float
__device__ __forceinline__ float df_val(dfloat d) { return d.hi + d.lo; }

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Max of non-negative v over each warp into the stripe of quantity q.
__device__ __forceinline__ void block_max(float v, double* acc, int q) {
    v = warp_max(v);
    if ((threadIdx.x & 31) == 0) {
        unsigned gw = (blockIdx.x * ((blockDim.x + 31) >> 5)) + (threadIdx.x >> 5);
        atomic_max_nonneg(acc + (gw & (kAccStripes - 1)) * kAccStride + q, (double)v);
    }
}

// ------------------------------------------------------------ complex
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// WA smoothing factors of gamma in float32: 1/gamma and log2(e)/gamma (the
// exponentials are exp2(t log2(e) / gamma)), the same on host and device.
__host__ __device__ inline void wa_scale(float gamma, float* inv_g, float* l2g) {
    *inv_g = 1.0f / gamma;
    *l2g = (float)(1.4426950408889634 / (double)gamma);
}

// -------------------------------------------------------- the context
struct Ctx {
    // problem
    int n = 0, logn = 0, m_mov = 0, m_fix = 0, E = 0;
    int64_t P = 0;
    double x0 = 0, y0 = 0, x1 = 0, y1 = 0, Lx = 0, Ly = 0, wb = 0, hb = 0, Ab = 0;
    double mov_area = 0;
    Grid grid{};
    fftpl_options opt{};
    int wa_max_degree = 0;

    // streams and events
    cudaStream_t stream = nullptr, side = nullptr, own_stream = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    bool profiling = false;
    double stage_ms[FFTPL_NUM_STAGES] = {};
    int64_t stage_launches[FFTPL_NUM_STAGES] = {};
    int64_t launches = 0;

    // device buffers
    float *w = nullptr, *h = nullptr, *fix_x = nullptr, *fix_y = nullptr;
    float *M = nullptr, *D = nullptr;
    long long* Dq = nullptr;
    float *T1 = nullptr, *PT = nullptr, *RT = nullptr;
    // tensor maps of T1, PT and RT (n/2 rows of n pairs; boxes of 4 pairs by
    // 256 rows, n/2 if smaller): the transposed tiles of the row and column
    // passes leave shared memory through the tensor-memory-access unit
    CUtensorMap map_t1{}, map_pt{}, map_rt{};
    bool spec_tma = false;      // the transposed stores go through the maps
    bool spec_maps_ok = false;  // the maps could be encoded
    float *psi = nullptr, *ex = nullptr, *ey = nullptr, *rho = nullptr;
    float2* E2 = nullptr;       // interleaved field (E_x, E_y) [n][n]
    float2 *tw = nullptr, *ph = nullptr;   // tables of the radix tensor-core path
    // pins re-laid into degree slabs (see k_wire.cu): slot base + 32 k + lane
    int4* slabs = nullptr;      // {base slot, degree, net count, lanes per net (0: one
                                // net per lane)}
    int nslabs = 0;
    int nbig = 0;               // the first nbig slabs: degree kBigMin..kBigMax
    int num_sms = 1;            // of the handle's device
    bool chain = false;         // launch_chain for the kernels being enqueued
    int64_t slab_slots = 0;
    int32_t *pin_cell = nullptr, *pin_slot = nullptr, *cell_pin_ptr = nullptr;
    float *pin_dx = nullptr, *pin_dy = nullptr;
    float2* gpin = nullptr;
    float2* gW2 = nullptr;      // interleaved wirelength gradient accumulator (m_mov),
                                // by internal number
    float2* pxy = nullptr;      // pin coordinates by slot, for the slabs of degree
                                // above kBigMax (their slots come first)
    float2* pos2 = nullptr;     // interleaved cell centres (m_mov), by internal number
    int32_t* cell_rank = nullptr;  // internal number of each movable cell (m_mov)
    // deterministic reductions: region 0 for the main stream, 1 for WA
    double* det_part = nullptr;
    unsigned* det_ticket = nullptr;
    int det_cap[2] = {0, 0};
    double* acc = nullptr;
    // what every evaluation starts from zero, in one block: the density map
    // (D or Dq), the FP64 sums, the wirelength gradient accumulator
    char* zero_block = nullptr;
    size_t zero_density = 0, zero_bytes = 0;   // bytes of the map, of the block
    int* err = nullptr;
    double* acc_host = nullptr;   // their totals in mapped host memory
    unsigned* report_count = nullptr;   // reports made, on the device
    unsigned reports = 0;               // reports enqueued

    // placement loop state (2 m_mov each: x then y)
    float *u = nullptr, *v = nullptr, *vprev = nullptr, *g = nullptr, *gprev = nullptr;
    float *gN = nullptr, *gW = nullptr;   // 2 m_mov each, loop scratch
    double* ctrl = nullptr;              // device control scalars
    double* recs = nullptr;              // device iteration records
    int recs_cap = 0;
    bool placing = false;
    int iter = 0;

    // host-side staging for fftpl_eval_host
    float *hx = nullptr, *hy = nullptr, *hg = nullptr;  // device staging (2m, 4m)

    // tensor-core solve path (solve_path FFTPL_SOLVE_TC_BF16X3), k_tc.cu
    struct TcPlan* tc = nullptr;
    // radix tensor-core path (solve_path FFTPL_SOLVE_TC_RADIX), k_tc.cu
    struct TcrPlan* tcr = nullptr;

    // captured CUDA graphs of fftpl_eval for one set of buffers, without and
    // with the report at the end: a caller that asks for the sums now and then
    // replays both (as one graph keyed by the report an evaluation of 1,000
    // cells, every second one with it, took 65 us on average instead of 17.7)
    struct EvalGraph {
        cudaGraphExec_t exec = nullptr;
        const void* key[8] = {};
        int64_t nkernels = 0;
    } eval_graph[2];
    // captured CUDA graph of one placement-loop iteration (fftpl_step), keyed
    // by the buffers its kernels take that can be reallocated
    cudaGraphExec_t loop_graph = nullptr;
    const void* loop_key[3] = {};
    int64_t loop_graph_nkernels = 0;
    // profiling ring of (stage, begin, end) event records
    std::vector<cudaEvent_t> prof_ev;
    std::vector<int> prof_stage;
    int prof_used = 0;

    bool rho_valid = false, fields_valid = false, split_valid = false;
    bool psi_valid = false;     // psi matches the current fields (it is formed on
                                // demand)
    bool own_capture = false;   // eval_impl is capturing
    bool replayed = false;      // a call went into a caller's own capture, whose
                                // replays the handle does not see: no map formed
                                // on demand counts as current from then on
    std::string last_error;
    std::vector<void*> dev_allocs;
    size_t dev_bytes = 0;
};

// Reduction descriptor of region r (0: main stream, 1: WA stream); atomics
// unless the handle is deterministic.
inline DetRed det_red(const Ctx& c, int r) {
    if (!c.det_part) return DetRed{nullptr, nullptr, 0};
    double* base = c.det_part + (r == 0 ? 0 : 2 * (size_t)c.det_cap[0]);
    return DetRed{base, c.det_ticket + r, c.det_cap[r]};
}

// Enqueues one placement-loop iteration on the handle's streams (no sync).
fftpl_status loop_enqueue(Ctx& c);
// One iteration replayed from the handle's loop graph (captured on first use
// when use_graphs is set); launch = false only captures it.
fftpl_status loop_iter(Ctx& c, bool launch);
// For the server (on a worker thread): start positions from host memory,
// loop initialisation, room for iters records and the loop graph; returns
// with the handle's stream idle.
fftpl_status serve_prepare(Ctx& c, const float* x0, const float* y0, int iters);
// Makes room for cap iteration records and numbers them from base_k.
fftpl_status loop_records(Ctx& c, int cap, double base_k);

// Sets the text fftpl_last_error(NULL) returns on this thread.
void set_global_error(const std::string& msg);

// Blocks of the cell kernels (one thread per cell up to kCellBlocks blocks per
// SM, striding beyond).
inline int cell_blocks(const Ctx& c) {
    const long long nb = ((long long)c.m_mov + kCellThreads - 1) / kCellThreads;
    const long long cap = (long long)c.num_sms * kCellBlocks;
    return (int)(nb < cap ? nb : cap);
}

// ------------------------------------------------------------ launchers
// (each returns the CUDA error of the launch)
void prepare_spectral(int logn);
// fixed cells into Dq (int64 units of 2^-32), at create
cudaError_t launch_scatter_fixed(Ctx& c, long long* Dq, cudaStream_t s);
// movable cells into the handle's D / Dq; write_pos: also the interleaved
// centres pos2 (by internal cell number) for the WA kernel; stage (2 m_mov
// floats or null): also a device copy of (x, y)
cudaError_t launch_scatter_mov(Ctx& c, const float* x, const float* y, bool write_pos,
                               float* stage, cudaStream_t s);
cudaError_t launch_bin_ranges(Ctx& c, const float* x, const float* y, int32_t* ranges,
                              cudaStream_t s);
cudaError_t launch_rows_fwd(Ctx& c, cudaStream_t s);
cudaError_t launch_cols_spectral(Ctx& c, cudaStream_t s);
cudaError_t launch_rows_inv(Ctx& c, cudaStream_t s);
// psi rows from PT (transform path; formed on demand, not in the evaluation);
// launch_rows_maps: psi, E_x and E_y into their separate maps
cudaError_t launch_rows_psi(Ctx& c, cudaStream_t s);
cudaError_t launch_rows_maps(Ctx& c, cudaStream_t s);
// Tensor maps for the transposed stores of the transform passes (host only,
// no allocation); clears c.spec_tma if the driver cannot encode them.
void spec_maps_init(Ctx& c);
// 2-D float32 tensor [rows][cols] in boxes of box_inner columns x box_outer rows.
bool make_map_f32(CUtensorMap* map, const float* base, int rows, int cols, int box_inner,
                  int box_outer);
cudaError_t launch_rho(Ctx& c, cudaStream_t s);
cudaError_t launch_split_field(Ctx& c, cudaStream_t s);
cudaError_t launch_q_to_f(const long long* q, float scale, float* out, int count, cudaStream_t s);
// scale (device double or null): multiplies the gradient written
cudaError_t launch_gather(Ctx& c, const float* x, const float* y, float* gx, float* gy,
                          bool adjoint, const double* scale, cudaStream_t s);
// interleave = false: pos2 already written (by launch_scatter_mov)
cudaError_t launch_wa_impl(Ctx& c, const float* x, const float* y, float gamma,
                           const float* scale_dev, const float* done, bool interleave,
                           cudaStream_t s);
cudaError_t launch_pin_sum(Ctx& c, float* gx, float* gy, bool few, bool chain, cudaStream_t s);
// 1 when the WA kernel runs slab pairs per warp (large instances)
int wa_pairs(const Ctx& c);
// blocks of the WA kernel: slabs of degree kBigMin..kBigMax, and the others
int wa_big_blocks(const Ctx& c);
int wa_small_blocks(const Ctx& c);

// create-time netlist layout (k_setup.cu): label rounds for the internal
// cell numbers (seeds every kSeedStride cells, kLabelRounds rounds, nets of
// more than kRankMaxDegree pins not followed), the orders of cells and nets,
// and the pin records in slab layout
constexpr int kSeedStride = 64;
constexpr int kLabelRounds = 6;
constexpr int kRankMaxDegree = 64;
cudaError_t launch_label_rounds(int m, int E, const int* np, const int* pc, int* lab, int* next,
                                int* dist, int* netlab, cudaStream_t s);
// ping-pong buffers of the radix sort: max(m, E) keys and values each,
// sort_counts of it counts
struct SortBuf {
    unsigned* key[2];
    int* val[2];
    int* counts;
};
size_t sort_counts(int n);
// internal cell numbers from the labels
cudaError_t launch_cell_rank(int m, const int* lab, const int* dist, SortBuf& buf, int* rank,
                             cudaStream_t s);
// buf.val[0]: the nets by descending degree (degrees below 2 last), then lowest
// cell number, then index
cudaError_t launch_net_order(int m, int E, int maxd, const int* np, const int* pc, const int* rank,
                             SortBuf& buf, cudaStream_t s);
cudaError_t launch_fill_slabs(int m, int nets, const int* order, const int2* by_degree,
                              const int* np, const int* pc, const float* dx, const float* dy,
                              const int* rank, const float* fix_x, const float* fix_y,
                              const int* cslot, int* spc, float* sdx, float* sdy, int* sslot,
                              cudaStream_t s);

// tensor-core solve path (k_tc.cu): tc_setup lays the plan out in a device
// block of tc_elems(n) bf16 elements owned by the handle and fills its
// cosine/sine tables on stream s; launch_tc part 0 splits rho (with the
// overflow and charge sums), 1 and 2 the forward contractions (2 with the
// spectral divide and the energy), 3 the inverse ones (E_x, E_y), 4 psi from
// the last solve.
size_t tc_elems(int n);
cudaError_t tc_setup(Ctx& c, uint16_t* block, cudaStream_t s);
void tc_free(Ctx& c);
cudaError_t launch_tc(Ctx& c, int part, cudaStream_t s);
cudaError_t tc_debug_gemm(const void* ah, const void* al, const void* bh, const void* bl, int M,
                          int N, int K, float* d, int nsplit, int no_loads, int* err,
                          cudaStream_t s);
// radix tensor-core path (k_tc.cu): tcr_setup lays the plan out in a device
// block of tcr_elems(n) bf16 elements and 2 n^2 float2 (Z, V) owned by the
// handle; launch_tcr part 0 the row pass, 1 the column pass, 2 the inverse
// row pass, 3 the overflow and charge sums alone.  launch_tcr_stage
// (k_spectral.cu): the pre- and post-processing kernels between its DFTs.
size_t tcr_elems(int n);
cudaError_t tcr_setup(Ctx& c, uint16_t* block, float2* zv, cudaStream_t s);
void tcr_free(Ctx& c);
cudaError_t launch_tcr(Ctx& c, int part, cudaStream_t s);
cudaError_t launch_tcr_stage(Ctx& c, int which, const float2* V, float2* Z, cudaStream_t s);
cudaError_t launch_cells(Ctx& c, const float* x, const float* y, float* gNx, float* gNy,
                         float* gWx, float* gWy, cudaStream_t s);
// placement loop
cudaError_t launch_loop_cells(Ctx& c, cudaStream_t s);
cudaError_t launch_loop_g(Ctx& c, cudaStream_t s);
cudaError_t launch_loop_update(Ctx& c, cudaStream_t s);
cudaError_t launch_place_init(Ctx& c, const float* x0, const float* y0, cudaStream_t s);
cudaError_t launch_gamma0(Ctx& c, cudaStream_t s);
// totals of the reported sums into c.acc_host (counted in c.reports); chain:
// the last operation enqueued on s is a kernel
cudaError_t launch_report(Ctx& c, bool chain, cudaStream_t s);
// N of the last solve to *out (device)
cudaError_t launch_energy_out(Ctx& c, double* out, cudaStream_t s);
// conjugate-gradient loop (k_step.cu)
cudaError_t launch_cg_g(Ctx& c, cudaStream_t s);
cudaError_t launch_cg_dir(Ctx& c, cudaStream_t s);
cudaError_t launch_cg_trial(Ctx& c, cudaStream_t s);
cudaError_t launch_cg_alpha(Ctx& c, cudaStream_t s);
cudaError_t launch_cg_update(Ctx& c, cudaStream_t s);

}  // namespace fftpl

// The opaque handle of the C ABI is the context.
struct fftpl_ctx : public fftpl::Ctx {};
