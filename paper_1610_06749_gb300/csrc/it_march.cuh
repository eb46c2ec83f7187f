// it_march.cuh -- the marches straight from L1/L2 (no shared-memory ring) of
// the single-grid and batched step kernels: one block of 128 columns of the
// flattened x-y plane over a chunk of z planes, and their tally reductions.
#pragma once

#include <cuda_runtime.h>

#include "it_device.cuh"
#include "it_internal.cuh"
#include "it_tma.cuh"

namespace itk {

constexpr int SK_THREADS = 128;
constexpr int SK_BLOCKS_F32 = 8, SK_BLOCKS_F64 = 6;   // resident blocks per SM
constexpr int DK_BLOCKS = 4;                            // of the direct kernel (128 registers)
constexpr double DK_LAT = 650.0, DK_THR = 190.0;        // its cycles per plane: alone, and per block it shares the SM with

// The direct march's units run in alternating order, step by step, where both
// sets of the state exceed this: a step then first reads what the step before
// it wrote last and is still in L2 (320x331x120, 203 MB: 47.3 to 45.6 us,
// 224x293x119, 125 MB: 30.0 to 29.6; smaller states stay in L2 either way and
// lose, 256x256x100, 105 MB: 22.8 to 23.6).
constexpr double DK_ALTERNATE = 115e6;

// CompSum's counterpart for FP64 states: a plain FP64 sum
struct PlainSum {
    double hi = 0.0;
    __device__ __forceinline__ void term(double x) { hi += x; }
    __device__ __forceinline__ void add(const PlainSum &o) { hi += o.hi; }
    __device__ __forceinline__ void scale(double w) { hi *= w; }
    __device__ __forceinline__ double value() const { return hi; }
    __device__ __forceinline__ PlainSum down(int o) const {
        PlainSum r;
        r.hi = __shfl_down_sync(0xffffffffu, hi, o);
        return r;
    }
};

template <typename T>
struct SumOf { using type = PlainSum; };
template <>
struct SumOf<float> { using type = CompSum; };

// the operations of add_sc, with the product kept for the tally
__device__ __forceinline__ float sk_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double sk_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sk_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double sk_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// Block sums of N values in a fixed order, added to tot[at ..]: value v is
// reduced by warp v mod 4 (four columns per lane, then shuffles) and
// converted to FP64 by its lane 0.
template <int N, typename Sum>
__device__ __forceinline__ void sk_reduce(const Sum (&v)[N], Sum (*buf)[SK_THREADS], double *tot, int at) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q) buf[q][tid] = v[q];
    __syncthreads();
#pragma unroll
    for (int q0 = 0; q0 < N; q0 += SK_THREADS / 32) {
        const int q = q0 + warp;
        if (q < N) {
            Sum s = buf[q][lane];
#pragma unroll
            for (int r = 1; r < SK_THREADS / 32; ++r) s.add(buf[q][lane + 32 * r]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s.add(s.down(o));
            if (lane == 0) tot[at + q] += s.value();
        }
    }
}

// Tally tid of a block's slot (at slots) from its sums (order: rec, lateral,
// space charge, anode from 5, cathode from 7), added or written.
template <bool PERIODIC, bool SC, int NV, typename T>
__device__ __forceinline__ void sk_slot(const double *tot, const Coef<T> &c, double *slots, int tid, int add) {
    double t = 0.0;
    if (tid == 0) t = tot[0] * c.rec_f;
    else if (tid < 3) t = tot[5 + tid - 1] * c.anode_f[tid - 1];
    else if (tid < 5) t = tot[7 + tid - 3] * c.cathode_f[tid - 3];
    // x and y weights are equal for dx = dy (latx_f == laty_f)
    else if (tid < 7) t = PERIODIC ? 0.0 : tot[1 + tid - 5] * c.latx_f[tid - 5];
    else t = SC ? tot[NV - 2 + tid - 7] * c.sc_f[tid - 7] : 0.0;
    double *sl = slots + tid;
    *sl = add ? *sl + t : t;
}

// Values a unit reduces: recombination, lateral +/- (absorbing), space charge +/-.
template <bool PERIODIC, bool SC>
struct MarchValues { static constexpr int N = 1 + (PERIODIC ? 0 : 2) + (SC ? 2 : 0); };
constexpr int MARCH_AN = 5, MARCH_CA = 7;   // electrode sums in a block's totals

// Column q0 + tid of the flattened plane over planes [k0, k1), one cell per
// thread, neighbours read through L1/L2 (step_simple_kernel).
template <typename T, typename Idx, bool PERIODIC, bool SC, class C>
__device__ __forceinline__ void simple_march(const T *__restrict__ ip, const T *__restrict__ im, T *__restrict__ op,
                                             T *__restrict__ om, int nx, int ny, int nz, Idx q0, int k0, int k1,
                                             const C &c, typename SumOf<T>::type (*buf)[SK_THREADS], double *tot) {
    using Sum = typename SumOf<T>::type;
    constexpr int NV = MarchValues<PERIODIC, SC>::N, AN = MARCH_AN, CA = MARCH_CA;
    const int tid = threadIdx.x;
    const Idx plane = (Idx)nx * (Idx)ny;
    Idx q = q0 + tid;
    const bool act = q < plane;
    if (!act) q = plane - 1;   // columns past the plane repeat the last one and store nothing
    const int j = (int)(q / (Idx)nx), i = (int)(q - (Idx)j * (Idx)nx);
    // neighbour columns (wrapped; absorbing faces hold zero instead)
    const Idx qxm = i > 0 ? q - 1 : q + (Idx)(nx - 1), qxp = i < nx - 1 ? q + 1 : q - (Idx)(nx - 1);
    const Idx qym = j > 0 ? q - (Idx)nx : q + (Idx)(ny - 1) * (Idx)nx;
    const Idx qyp = j < ny - 1 ? q + (Idx)nx : q - (Idx)(ny - 1) * (Idx)nx;
    const bool hxm = PERIODIC || i > 0, hxp = PERIODIC || i < nx - 1;
    const bool hym = PERIODIC || j > 0, hyp = PERIODIC || j < ny - 1;
    Sum v[NV];
    Idx base = (Idx)k0 * plane;
    T zm[2], n[2];
    T zp[2];   // loaded one plane ahead
    zm[0] = k0 > 0 ? ip[base - plane + q] : T(0);
    zm[1] = k0 > 0 ? im[base - plane + q] : T(0);
    n[0] = ip[base + q];
    n[1] = im[base + q];
    zp[0] = k0 + 1 < nz ? ip[base + plane + q] : T(0);
    zp[1] = k0 + 1 < nz ? im[base + plane + q] : T(0);
    const int sides = (i == 0) + (i == nx - 1) + (j == 0) + (j == ny - 1);
    const T first[2] = {n[0], n[1]};   // the chunk's first plane (anode tally)
    T last[2] = {n[0], n[1]};
#pragma unroll 2
    for (int k = k0; k < k1; ++k, base += plane) {
        const T rr = n[0] * n[1];
        T z2[2], w[2];
        const bool more = k + 1 < k1 && k + 2 < nz;
        z2[0] = more ? ip[base + 2 * plane + q] : T(0);
        z2[1] = more ? im[base + 2 * plane + q] : T(0);
        const T d = SC ? n[0] - n[1] : T(0);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const T *in = s ? im : ip;
            const T xm = hxm ? in[base + qxm] : T(0), xp = hxp ? in[base + qxp] : T(0);
            const T ym = hym ? in[base + qym] : T(0), yp = hyp ? in[base + qyp] : T(0);
            w[s] = upd7(n[s], xm, xp, ym, yp, zm[s], zp[s], rr, c.wx[s], c.wzm[s], c.wzp[s], c.adt);
            if constexpr (SC) {
                const T t = sk_mul(n[s], d);
                w[s] = sk_fma(c.sc[s], t, w[s]);
                v[NV - 2 + s].term(t);
            }
            if constexpr (!PERIODIC) {
                if (sides > 0) v[1 + s].term(n[s]);
            }
        }
        v[0].term(rr);
        if (act) {
            op[base + q] = w[0];
            om[base + q] = w[1];
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            last[s] = n[s];
            zm[s] = n[s];
            n[s] = zp[s];
            zp[s] = z2[s];
        }
    }
    // lateral faces: what leaves through the x and y sides of this column
    if constexpr (!PERIODIC) {
        v[1].scale((T)sides);
        v[2].scale((T)sides);
    }
    if (!act) {
#pragma unroll
        for (int t = 0; t < NV; ++t) v[t] = Sum{};
    }
    sk_reduce<NV>(v, buf, tot, 0);
    if (k0 == 0) {
        Sum e[2];
        if (act) { e[0].term(first[0]); e[1].term(first[1]); }
        sk_reduce<2>(e, buf, tot, AN);
    }
    if (k1 == nz) {
        Sum e[2];
        if (act) { e[0].term(last[0]); e[1].term(last[1]); }
        sk_reduce<2>(e, buf, tot, CA);
    }
}

// One thread's sum of a tally over its float4 segments.
template <bool EXACT>
struct QuadSum {   // four cells in plain FP32, then compensated
    CompSum c;
    __device__ __forceinline__ void add(float2 a, float2 b) {
        c.term(__fadd_rn(__fadd_rn(a.x, a.y), __fadd_rn(b.x, b.y)));
    }
    __device__ __forceinline__ CompSum total() const { return c; }
};
template <>
struct QuadSum<true> {   // every cell compensated
    CompSum2 c;
    __device__ __forceinline__ void add(float2 a, float2 b) {
        c.term(a);
        c.term(b);
    }
    __device__ __forceinline__ CompSum total() const { return c.total(); }
};

// The same with a float4 x-segment per thread (nx % 4 == 0), segment q0 + tid
// (step_direct_kernel).  Every cell's terms enter compensated sums, so the
// tallies are as close as the simple kernel's; in paired instructions that
// costs nothing against four cells added in FP32 first (128x128x200 9.8 us per
// step both ways).  With space charge there are three such sums and it does
// (384x320x128 54.5 us against 53.4, 128x128x200 12.2 against 11.4, 256x256x100
// 24.6 against 23.4): there only EXACT instances sum so, for the widths whose
// tallies the simple kernel would otherwise sum (exact_sums).
template <typename Idx, bool PERIODIC, bool SC, bool EXACT, class C>
__device__ __forceinline__ void direct_march(const float *__restrict__ ip, const float *__restrict__ im,
                                             float *__restrict__ op, float *__restrict__ om, int nx, int ny, int nz,
                                             Idx q0, int k0, int k1, const C &c, CompSum (*buf)[SK_THREADS],
                                             double *tot) {
    constexpr int NV = MarchValues<PERIODIC, SC>::N, AN = MARCH_AN, CA = MARCH_CA;
    const int tid = threadIdx.x, lane = tid & 31;
    const unsigned ncol4 = (unsigned)nx >> 2;
    const Idx plane = (Idx)nx * (Idx)ny, plane4 = (Idx)ncol4 * (Idx)ny;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    Idx q4 = q0 + tid;
    const bool act = q4 < plane4;
    if (!act) q4 = plane4 - 1;   // segments past the plane repeat the last one and store nothing
    const int j = (int)(q4 / (Idx)ncol4), c4 = (int)(q4 - (Idx)j * (Idx)ncol4);
    const Idx q = 4 * q4;
    const bool first = c4 == 0, last = c4 == (int)ncol4 - 1;
    const Idx qu = j > 0 ? q - (Idx)nx : q + (Idx)(ny - 1) * (Idx)nx;
    const Idx qd = j < ny - 1 ? q + (Idx)nx : q - (Idx)(ny - 1) * (Idx)nx;
    const bool hu = PERIODIC || j > 0, hd = PERIODIC || j < ny - 1;
    const bool el = lane == 0 || first, er = lane == 31 || last || q4 + 1 >= plane4;
    const Idx ql = first ? q + (Idx)(nx - 1) : q - 1, qr = last ? q - (Idx)(nx - 4) : q + 4;
    CompSum v[NV];
    QuadSum<!SC || EXACT> rec, spc[2];   // recombination, space charge
    Idx base = (Idx)k0 * plane;
    auto ld = [&](const float *f, Idx e) { return __ldg(reinterpret_cast<const float4 *>(f + e)); };
    float4 zm[2], n[2], zp[2];
    zm[0] = k0 > 0 ? ld(ip, base - plane + q) : zero4;
    zm[1] = k0 > 0 ? ld(im, base - plane + q) : zero4;
    n[0] = ld(ip, base + q);
    n[1] = ld(im, base + q);
    zp[0] = k0 + 1 < nz ? ld(ip, base + plane + q) : zero4;
    zp[1] = k0 + 1 < nz ? ld(im, base + plane + q) : zero4;
    CompSum an[2];   // the chunk's first plane (anode tally)
    add4(an[0], n[0]);
    add4(an[1], n[1]);
    // y neighbours and the x neighbours a shuffle cannot give, of plane k
    float4 up[2], dn[2];
    float le[2], re[2];
    auto around = [&](Idx at) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const float *in = s ? im : ip;
            up[s] = hu ? ld(in, at + qu) : zero4;
            dn[s] = hd ? ld(in, at + qd) : zero4;
            le[s] = el && (PERIODIC || !first) ? __ldg(in + at + ql) : 0.f;
            re[s] = er && (PERIODIC || !last) ? __ldg(in + at + qr) : 0.f;
        }
    };
    around(base);
    for (int k = k0; k < k1; ++k, base += plane) {
        float4 z2[2];   // two planes above, for the next round
        const bool more = k + 1 < k1 && k + 2 < nz;
        z2[0] = more ? ld(ip, base + 2 * plane + q) : zero4;
        z2[1] = more ? ld(im, base + 2 * plane + q) : zero4;
        const float2 rxy = __fmul2_rn(make_float2(n[0].x, n[0].y), make_float2(n[1].x, n[1].y));
        const float2 rzw = __fmul2_rn(make_float2(n[0].z, n[0].w), make_float2(n[1].z, n[1].w));
        float2 dxy, dzw;
        if (SC) sc_diff4(n[0], n[1], dxy, dzw);
        float4 w4[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            float l = __shfl_up_sync(0xffffffffu, n[s].w, 1);
            float r = __shfl_down_sync(0xffffffffu, n[s].x, 1);
            if (el) l = le[s];
            if (er) r = re[s];
            w4[s] = upd7x4(n[s], l, r, up[s], dn[s], zm[s], zp[s], rxy, rzw, c.wx[s], c.wzm[s], c.wzp[s], c.adt);
            if constexpr (SC) {
                float2 pxy, pzw;
                w4[s] = add_sc4(w4[s], c.sc[s], n[s], dxy, dzw, pxy, pzw);
                spc[s].add(pxy, pzw);
            }
            if constexpr (!PERIODIC) {
                if (first) v[1 + s].term(n[s].x);
                if (last) v[1 + s].term(n[s].w);
                if (j == 0) add4(v[1 + s], n[s]);
                if (j == ny - 1) add4(v[1 + s], n[s]);
            }
        }
        if (k + 1 < k1) around(base + plane);
#pragma unroll
        for (int s = 0; s < 2; ++s)
            if (act) *reinterpret_cast<float4 *>((s ? om : op) + base + q) = w4[s];
        rec.add(rxy, rzw);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            zm[s] = n[s];
            n[s] = zp[s];
            zp[s] = z2[s];
        }
    }
    v[0] = rec.total();
    if constexpr (SC) {
        v[NV - 2] = spc[0].total();
        v[NV - 1] = spc[1].total();
    }
    if (!act) {
#pragma unroll
        for (int t = 0; t < NV; ++t) v[t] = CompSum{};
        an[0] = an[1] = CompSum{};
    }
    sk_reduce<NV>(v, buf, tot, 0);
    if (k0 == 0) sk_reduce<2>(an, buf, tot, AN);
    if (k1 == nz) {
        CompSum e[2];
        if (act) { add4(e[0], zm[0]); add4(e[1], zm[1]); }   // the last plane (cathode tally)
        sk_reduce<2>(e, buf, tot, CA);
    }
}

}  // namespace itk
