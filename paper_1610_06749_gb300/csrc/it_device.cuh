// it_device.cuh -- device helpers shared by the kernel files.
#pragma once

#include <cuda_runtime.h>

namespace itk {

// ---------------------------------------------------------------------------
// deterministic block reduction of N doubles (fixed shuffle and warp order)
// ---------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N], double *smem /* [32][N] */) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < N; ++q) smem[warp * N + q] = v[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        for (int q = 0; q < N; ++q) {
            double s = 0.0;
            for (int w = 0; w < nw; ++w) s += smem[w * N + q];
            v[q] = s;
        }
    }
}

// Sum of quantity q of n records of `width` doubles by one warp, in a fixed
// order: lane l adds records l, l + 32, ..., then the shuffle tree (the sum
// is lane 0's).
__device__ __forceinline__ double warp_strided_sum(const double *__restrict__ v, int n, int q, int width, int lane) {
    double t = 0.0;
    for (int b = lane; b < n; b += 32) t += v[(size_t)b * width + q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    return t;
}

// FP32 sum that carries the rounding error of each addition (Knuth's
// two-sum), so a sum of some hundred terms keeps about 46 bits: as good as
// FP64 for terms that are FP32 products.  Its terms are kept times 2^-32,
// which costs nothing (the products with it are exact, in fused
// multiply-adds), so that no sum of fewer than 2^32 finite terms overflows as
// an FP64 one would not; terms below 2^-94 lose bits of less than 2^-117.  A
// sum that meets an infinity or a NaN is returned as it is.
constexpr float SUM_SCALE = 0x1p-32f;
constexpr double SUM_UNSCALE = 0x1p32;

struct CompSum {
    float hi = 0.f, lo = 0.f;   // times SUM_SCALE
    __device__ __forceinline__ void term(float x) {
        const float s = __fmaf_rn(x, SUM_SCALE, hi);
        const float b = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fmaf_rn(x, SUM_SCALE, -b)));
        hi = s;
    }
    __device__ __forceinline__ void add(float x) {   // x scaled already
        const float s = __fadd_rn(hi, x);
        const float b = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
        hi = s;
    }
    __device__ __forceinline__ void add(const CompSum &o) {
        const float l = o.lo;
        add(o.hi);
        lo = __fadd_rn(lo, l);
    }
    __device__ __forceinline__ void scale(float w) {   // w a small whole number
        const float p = __fmul_rn(hi, w);
        lo = __fmaf_rn(lo, w, __fmaf_rn(hi, w, -p));
        hi = p;
    }
    __device__ __forceinline__ double value() const {
        return (isfinite(hi) ? (double)hi + (double)lo : (double)hi) * SUM_UNSCALE;
    }
    __device__ __forceinline__ CompSum down(int o) const {
        CompSum r;
        r.hi = __shfl_down_sync(0xffffffffu, hi, o);
        r.lo = __shfl_down_sync(0xffffffffu, lo, o);
        return r;
    }
};

__device__ __forceinline__ void add4(CompSum &c, float4 v) { c.term(v.x); c.term(v.y); c.term(v.z); c.term(v.w); }

// Two such sums side by side in paired-FP32 instructions (seven for two terms;
// multiplications by -1 are exact, so every line is one rounding as above).
struct CompSum2 {
    float2 hi = make_float2(0.f, 0.f), lo = make_float2(0.f, 0.f);
    __device__ __forceinline__ void term(float2 x) {
        const float2 neg = make_float2(-1.f, -1.f), sc = make_float2(SUM_SCALE, SUM_SCALE);
        const float2 s = __ffma2_rn(x, sc, hi);
        const float2 nb = __ffma2_rn(s, neg, hi);                      // hi - s
        const float2 eh = __ffma2_rn(__fadd2_rn(s, nb), neg, hi);      // hi - (s - b)
        lo = __fadd2_rn(lo, __fadd2_rn(eh, __ffma2_rn(x, sc, nb)));
        hi = s;
    }
    __device__ __forceinline__ CompSum total() const {
        CompSum t;
        t.add(hi.x);
        t.add(hi.y);
        t.lo = __fadd_rn(t.lo, __fadd_rn(lo.x, lo.y));
        return t;
    }
};

// One cell of the update as an increment in flux form:
//   n + [wd ((l + r) + (u + d) - 4 n) + wzm (zm - n) + wzp (zp - n) - adt rr]
// (wd = wx = wy: the cells are cubes).  Every transport term is a weight
// times a neighbour-minus-cell difference, so the transport part of the
// bracket sums to zero over the grid whatever the rounded weights: charge
// is moved, never made or lost, and each weight is simply its nearest FP32
// value.  The bracket's terms are small next to n, so their rounding errors
// are too; the one rounding of n + bracket is the only one at the scale of
// n.  The same operation sequence in every kernel, so all kernels round
// identically.
__device__ __forceinline__ float upd7(float n, float l, float r, float u, float d, float zm, float zp, float rr,
                                      float wd, float wzm, float wzp, float adt) {
    const float s4 = __fadd_rn(__fadd_rn(l, r), __fadd_rn(u, d));
    float v = __fmul_rn(wd, __fmaf_rn(-4.f, n, s4));
    v = __fmaf_rn(wzm, __fsub_rn(zm, n), v);
    v = __fmaf_rn(wzp, __fsub_rn(zp, n), v);
    v = __fmaf_rn(-adt, rr, v);
    return __fadd_rn(n, v);
}

__device__ __forceinline__ double upd7(double n, double l, double r, double u, double d, double zm, double zp,
                                       double rr, double wd, double wzm, double wzp, double adt) {
    const double s4 = __dadd_rn(__dadd_rn(l, r), __dadd_rn(u, d));
    double v = __dmul_rn(wd, __fma_rn(-4.0, n, s4));
    v = __fma_rn(wzm, __dsub_rn(zm, n), v);
    v = __fma_rn(wzp, __dsub_rn(zp, n), v);
    v = __fma_rn(-adt, rr, v);
    return __dadd_rn(n, v);
}

// The space-charge term of one cell, after upd7: v + sc n (n+ - n-), in this
// operation order in every kernel (the paired form is add_sc4).
__device__ __forceinline__ float add_sc(float v, float sc, float n, float p, float m) {
    return __fmaf_rn(sc, __fmul_rn(n, __fsub_rn(p, m)), v);
}
__device__ __forceinline__ double add_sc(double v, double sc, double n, double p, double m) {
    return __fma_rn(sc, __dmul_rn(n, __dsub_rn(p, m)), v);
}

}  // namespace itk
