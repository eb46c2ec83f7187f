// it_kernels.cu -- deposition, the simple step kernel, monitor and tally
// reduction kernels.
//
// Deposition follows Eqs. (linear_density), (Gaussian), (created): a track
// parallel to E with N0 = LET/W ions per cm and radial profile
// N0/(pi b^2) exp(-r^2/b^2), integrated over each cell, identical on every z
// plane.  The step is the Appendix scheme (Lax-Wendroff drift along z, FTCS
// diffusion on three axes, -alpha n+ n- from the old level), written in flux
// form so the tallies of what crosses the electrode faces close the charge
// balance.
#include <algorithm>
#include <cmath>

#include "it_device.cuh"
#include "it_internal.cuh"
#include "it_march.cuh"

namespace itk {

// ---------------------------------------------------------------------------
// simple step: any grid and type, neighbours read through L1/L2
// ---------------------------------------------------------------------------
// A thread owns one column of the flattened x-y plane (cell q of nx ny) and
// marches it over a chunk of z planes, so the z neighbours stay in registers
// and the cell's position costs one division per chunk; a block is 128
// neighbouring columns, whatever nx is.
//
// What bounds it: FP64 states run at the FP64 rate of this GPU (two lanes per
// SM and clock: 24 operations per cell are 10 us of a 48x48x100 step), FP32
// states at the L1 wavefronts of ten scalar loads and two stores per cell.
// The tallies therefore stay off the FP64 pipe: FP32 states sum in FP32 with
// the rounding error of every addition carried along (CompSum), the block
// reduction runs in the same form and one lane converts its result; faces
// (electrodes, absorbing sides) are only reduced by blocks that touch them.
// With one cell per thread, an FP64 addition per cell and a nine-value FP64
// shuffle reduction per warp, the earlier form took 49 us per step on
// 48x48x100 in FP64 and 224 us on 301x173x97 in FP32; this one takes 16.2
// and 31 us.  Eight blocks per SM (64 registers) with the plane above loaded
// one plane ahead: ten blocks without that took 34.6 us on 301x173x97.
// Work unit u: column block u mod npb, z chunk u / npb of nchunk.  A block
// takes units blockIdx.x, blockIdx.x + gridDim.x, ...; its tally slot is
// added to (add = 1) or replaced (add = 0).
template <typename T, typename Idx, bool PERIODIC, bool SC>
__global__ void __launch_bounds__(SK_THREADS, (sizeof(T) == 4 ? SK_BLOCKS_F32 : SK_BLOCKS_F64))
step_simple_kernel(const T *__restrict__ ip, const T *__restrict__ im, T *__restrict__ op, T *__restrict__ om, int nx,
                   int ny, int nz, unsigned npb, unsigned nchunk, const Coef<T> c, double *__restrict__ slots,
                   int add) {
    using Sum = typename SumOf<T>::type;
    constexpr int NV = MarchValues<PERIODIC, SC>::N;
    __shared__ double raw[5 * SK_THREADS];
    Sum(*buf)[SK_THREADS] = reinterpret_cast<Sum(*)[SK_THREADS]>(raw);
    static_assert(sizeof(Sum) == sizeof(double), "reduction scratch");
    __shared__ double tot[9];
    const int tid = threadIdx.x;
    if (tid < 9) tot[tid] = 0.0;
    const unsigned long long units = (unsigned long long)npb * nchunk;
    for (unsigned long long u = blockIdx.x; u < units; u += gridDim.x) {
        const unsigned pb = (unsigned)(u % npb), ch = (unsigned)(u / npb);
        const int k0 = (int)((long long)nz * ch / nchunk), k1 = (int)((long long)nz * (ch + 1) / nchunk);
        simple_march<T, Idx, PERIODIC, SC>(ip, im, op, om, nx, ny, nz, (Idx)pb * SK_THREADS, k0, k1, c, buf, tot);
    }
    __syncthreads();
    if (tid < 9) sk_slot<PERIODIC, SC, NV>(tot, c, slots + (size_t)blockIdx.x * NT, tid, add);
}

// Chunks per column and blocks of a launch, by the fitted time of a split.
// FP64: the FP64 pipe of an SM works off its units one after another, 2300
// cycles per plane of a unit and 0.45 planes for a unit's start and
// reduction; a single block per SM leaves it a tenth idle.  FP32: a resident
// block takes 600 cycles per plane plus 75 for every block it shares the SM
// with, each round of units starts with two planes of loads.  (48x48x100 in
// FP64: 16.2 us at 25 chunks, 17.7 at 8, 116 at one; 301x173x97 in FP32
// 30.7-33 us at 2 to 9 chunks, 37.9 at 20; 200x111x280 28.0 us at 6, 54 at
// 2, 32 at 40.)
struct SkShape { unsigned npb, nchunk, grid; };
static SkShape sk_shape(int nx, int ny, int nz, bool fp64) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const unsigned long long plane = (unsigned long long)nx * ny;
    const unsigned long long npb = (plane + SK_THREADS - 1) / SK_THREADS;
    const unsigned long long resident = std::min<unsigned long long>(
        (unsigned long long)sms * (fp64 ? SK_BLOCKS_F64 : SK_BLOCKS_F32), IT_NOALLOC_MAX_BLOCKS);
    unsigned best = 1;
    double best_cost = 1e300;
    for (unsigned c = 1; c <= (unsigned)nz; c += std::max(1u, c / 16)) {   // a few hundred splits at most
        const unsigned long long units = npb * c;
        if (c > 1 && units > 8 * resident) break;
        const double kc = (nz + c - 1) / c;
        double cost;
        if (fp64) {
            const double per_sm = (double)((units + sms - 1) / sms);
            cost = per_sm * (kc + 0.45) * 2300.0 * (per_sm == 1.0 ? 1.1 : 1.0) + (kc + 2.0) * 300.0;
        } else {
            const unsigned long long rem = units % resident;
            cost = (double)(units / resident) * (kc + 2.0) * (600.0 + 75.0 * SK_BLOCKS_F32);
            if (rem) cost += (kc + 2.0) * (600.0 + 75.0 * (double)((rem + sms - 1) / sms));
        }
        if (cost < 0.99 * best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    const unsigned long long units = npb * best;
    return SkShape{(unsigned)npb, best, (unsigned)std::min(units, resident)};
}

int simple_grid(const it_ctx *c) { return (int)sk_shape(c->g.nx, c->g.ny, c->g.nz, c->prec == IT_FP64).grid; }

int simple_grid_f32(int nx, int ny, int nz) { return (int)sk_shape(nx, ny, nz, false).grid; }

template <typename T>
static int sk_launch(const T *ip, const T *im, T *op, T *om, int nx, int ny, int nz, const Coef<T> &cf, bool periodic,
                     double *slots, int add, cudaStream_t s) {
    const SkShape h = sk_shape(nx, ny, nz, sizeof(T) == 8);
    // 32-bit element offsets where they reach (a neighbour plane beyond the
    // last is never formed: its load is predicated off, its offset may wrap)
    const bool small = (unsigned long long)nx * ny * nz <= 0xffffffffull - 2 * SK_THREADS;
    const bool sc = cf.sc_on != 0;
    auto go = [&](auto *k) { k<<<h.grid, SK_THREADS, 0, s>>>(ip, im, op, om, nx, ny, nz, h.npb, h.nchunk, cf, slots, add); };
    if (small) {
        if (periodic) sc ? go(step_simple_kernel<T, uint32_t, true, true>) : go(step_simple_kernel<T, uint32_t, true, false>);
        else sc ? go(step_simple_kernel<T, uint32_t, false, true>) : go(step_simple_kernel<T, uint32_t, false, false>);
    } else {
        if (periodic) sc ? go(step_simple_kernel<T, uint64_t, true, true>) : go(step_simple_kernel<T, uint64_t, true, false>);
        else sc ? go(step_simple_kernel<T, uint64_t, false, true>) : go(step_simple_kernel<T, uint64_t, false, false>);
    }
    IT_CK(cudaGetLastError());
    return IT_OK;
}

int launch_step_simple(it_ctx *c, cudaStream_t s) {
    const int cur = c->cur, nxt = cur ^ 1;
    const bool per = c->p.lateral_bc == IT_PERIODIC;
    const int rc = c->prec == IT_FP32
                       ? sk_launch<float>((const float *)c->n[cur][0], (const float *)c->n[cur][1],
                                          (float *)c->n[nxt][0], (float *)c->n[nxt][1], c->g.nx, c->g.ny, c->g.nz,
                                          c->cf, per, c->d_slots, 1, s)
                       : sk_launch<double>((const double *)c->n[cur][0], (const double *)c->n[cur][1],
                                           (double *)c->n[nxt][0], (double *)c->n[nxt][1], c->g.nx, c->g.ny, c->g.nz,
                                           c->cd, per, c->d_slots, 1, s);
    if (rc) return rc;
    c->cur = nxt;
    return IT_OK;
}

// The simple step on caller-given FP32 arrays; writes (not adds) the tallies
// of simple_grid_f32(nx, ny, nz) slots of NT doubles.
int launch_step_simple_raw_f32(const float *ip, const float *im, float *op, float *om, int nx, int ny, int nz,
                               const Coef<float> &cf, bool periodic, double *slots, cudaStream_t s) {
    return sk_launch<float>(ip, im, op, om, nx, ny, nz, cf, periodic, slots, 0, s);
}

// ---------------------------------------------------------------------------
// direct march: FP32, nx % 4 == 0, columns of float4 straight from L1/L2
// ---------------------------------------------------------------------------
// The simple kernel's work split with a float4 x-segment per thread and the
// paired-FP32 update: a block is 128 neighbouring segments of the flattened
// x-y plane, marched over a chunk of planes.  x neighbours come by warp
// shuffle (a load at the ends of a warp or row), y neighbours by 16-byte
// loads that mostly hit L1, the plane above is loaded one plane ahead.
// It has no ring to fill and no slot hand-back, which is what a step of a
// small or middle-sized grid (state in L2) spends its time on with the
// TMA-staged kernel; on grids that stream from HBM the ring wins.
// 128x128x200 9.9-12.4 us per step against 19.6 with the ring, 256x256x100
// 22.8 against a fitted 24.6; 256x256x400 86 against 70.
template <typename Idx, bool PERIODIC, bool SC, bool EXACT>
__global__ void __launch_bounds__(SK_THREADS, DK_BLOCKS)
step_direct_kernel(const float *__restrict__ ip, const float *__restrict__ im, float *__restrict__ op,
                   float *__restrict__ om, int nx, int ny, int nz, unsigned npb, unsigned nchunk, int rev,
                   const Coef<float> c, double *__restrict__ slots) {
    constexpr int NV = MarchValues<PERIODIC, SC>::N;
    __shared__ double raw[5 * SK_THREADS];
    CompSum(*buf)[SK_THREADS] = reinterpret_cast<CompSum(*)[SK_THREADS]>(raw);
    __shared__ double tot[9];
    const int tid = threadIdx.x;
    if (tid < 9) tot[tid] = 0.0;
    const unsigned long long units = (unsigned long long)npb * nchunk;
    for (unsigned long long q = blockIdx.x; q < units; q += gridDim.x) {
        const unsigned long long u = rev ? units - 1 - q : q;
        const unsigned pb = (unsigned)(u % npb), ch = (unsigned)(u / npb);
        const int k0 = (int)((long long)nz * ch / nchunk), k1 = (int)((long long)nz * (ch + 1) / nchunk);
        direct_march<Idx, PERIODIC, SC, EXACT>(ip, im, op, om, nx, ny, nz, (Idx)pb * SK_THREADS, k0, k1, c, buf, tot);
    }
    __syncthreads();
    if (tid < 9) sk_slot<PERIODIC, SC, NV>(tot, c, slots + (size_t)blockIdx.x * NT, tid, 1);
}

// Chunks and blocks, fitted as the simple kernel's are; *cycles receives the
// fitted time.
static SkShape dk_shape(int nx, int ny, int nz, double *cycles = nullptr) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const unsigned long long npb = ((unsigned long long)(nx / 4) * ny + SK_THREADS - 1) / SK_THREADS;
    const unsigned long long resident = (unsigned long long)sms * DK_BLOCKS;
    unsigned best = 1;
    double best_cost = 1e300;
    for (unsigned c = 1; c <= (unsigned)nz; c += std::max(1u, c / 16)) {
        const unsigned long long units = npb * c;
        if (c > 1 && units > 8 * resident) break;
        const double kc = (nz + c - 1) / c;
        const unsigned long long rem = units % resident;
        double cost = (double)(units / resident) * (kc + 2.0) * (DK_LAT + DK_THR * DK_BLOCKS);
        if (rem) cost += (kc + 2.0) * (DK_LAT + DK_THR * (double)((rem + sms - 1) / sms));
        if (cost < 0.99 * best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    if (cycles) *cycles = best_cost;
    const unsigned long long units = npb * best;
    return SkShape{(unsigned)npb, best, (unsigned)std::min(units, resident)};
}

int direct_grid(const it_ctx *c) {
    if (c->prec != IT_FP32 || c->g.nx % 4 != 0) return 0;
    return (int)dk_shape(c->g.nx, c->g.ny, c->g.nz).grid;
}

// Fitted time of a direct step in us: its rounds at 1.9 GHz and a launch, or,
// when both sets of the state outgrow L2, 1.45 times a copy at 6.8 TB/s.
double direct_us(const it_ctx *c) {
    double cycles = 0.0;
    (void)dk_shape(c->g.nx, c->g.ny, c->g.nz, &cycles);
    const double bytes = 16.0 * (double)c->g.cells();
    return std::max(cycles / 1900.0 + 1.5, bytes > 100e6 ? 1.45 * bytes / 6.8e6 : 0.0);
}

int launch_step_direct(it_ctx *c, cudaStream_t s) {
    const int cur = c->cur, nxt = cur ^ 1;
    const int nx = c->g.nx, ny = c->g.ny, nz = c->g.nz;
    const SkShape h = dk_shape(nx, ny, nz);
    const int rev = cur != c->base && 16.0 * (double)c->g.cells() > DK_ALTERNATE;
    const float *ip = (const float *)c->n[cur][0], *im = (const float *)c->n[cur][1];
    float *op = (float *)c->n[nxt][0], *om = (float *)c->n[nxt][1];
    auto go = [&](auto *k) { k<<<h.grid, SK_THREADS, 0, s>>>(ip, im, op, om, nx, ny, nz, h.npb, h.nchunk, rev, c->cf, c->d_slots); };
    // 32-bit element offsets: the z-march family takes grids below 2^32 cells
    const bool exact = exact_sums(nx);
    if (c->p.lateral_bc == IT_PERIODIC)
        !c->cf.sc_on ? go(step_direct_kernel<uint32_t, true, false, true>)
        : exact      ? go(step_direct_kernel<uint32_t, true, true, true>)
                     : go(step_direct_kernel<uint32_t, true, true, false>);
    else
        !c->cf.sc_on ? go(step_direct_kernel<uint32_t, false, false, true>)
        : exact      ? go(step_direct_kernel<uint32_t, false, true, true>)
                     : go(step_direct_kernel<uint32_t, false, true, false>);
    IT_CK(cudaGetLastError());
    c->cur = nxt;
    return IT_OK;
}

// ---------------------------------------------------------------------------
// monitor: in-domain ions and extreme densities of the current state
// ---------------------------------------------------------------------------
// Per-thread accumulation of one cell of each species into T partial sums
// and extremes; the partials are moved to FP64 by flush(), which callers run
// once per at most 32 cells outside the per-cell code (FP64 is slow on this
// GPU: an FP64 add in the per-cell path, even a predicated one, would bound
// the kernel).
template <typename T>
struct MonAcc {
    double sum[2] = {0.0, 0.0};
    T part[2] = {0, 0};
    T mn[2] = {(T)INFINITY, (T)INFINITY}, mx[2] = {(T)-INFINITY, (T)-INFINITY};
    __device__ __forceinline__ void add(T a, T b) {
        part[0] += a; part[1] += b;          // a NaN propagates into the sums
        mn[0] = a < mn[0] ? a : mn[0]; mn[1] = b < mn[1] ? b : mn[1];
        mx[0] = a > mx[0] ? a : mx[0]; mx[1] = b > mx[1] ? b : mx[1];
    }
    __device__ __forceinline__ void flush() {
        sum[0] += (double)part[0]; sum[1] += (double)part[1];
        part[0] = part[1] = 0;
    }
};

// In-domain sums and extremes of both species, one row of NM values per CTA.
// FP32 states on 16-byte boundaries are read as float4, four loads of each
// species in flight per thread, and summed in FP32 over 32 cells (two
// rounds of four float4) before FP64; other cells are read one by one and
// summed in T over up to 32 cells.
template <typename T>
__global__ void __launch_bounds__(256)
monitor_kernel(const T *__restrict__ ip, const T *__restrict__ im, size_t total, double vol,
               double *__restrict__ mon) {
    __shared__ double bsum[2][256];
    __shared__ T bext[4][256];
    MonAcc<T> acc;
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t nthr = (size_t)gridDim.x * blockDim.x;
    size_t done = 0;
    const bool vec = sizeof(T) == 4 && (((uintptr_t)ip | (uintptr_t)im) & 15) == 0;
    if (vec) {
        const size_t n4 = total / 4;
        const float4 *p4 = reinterpret_cast<const float4 *>(ip);
        const float4 *m4 = reinterpret_cast<const float4 *>(im);
        size_t q = tid;
        bool more = true;
        while (more) {
            // one round: up to two groups of four float4 per species (32 cells)
            for (int g = 0; g < 2; ++g) {
                if (q + 3 * nthr >= n4) { more = false; break; }
                float4 a[4], b[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    a[u] = __ldcs(p4 + q + u * nthr);
                    b[u] = __ldcs(m4 + q + u * nthr);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    acc.add(a[u].x, b[u].x); acc.add(a[u].y, b[u].y);
                    acc.add(a[u].z, b[u].z); acc.add(a[u].w, b[u].w);
                }
                q += 4 * nthr;
            }
            acc.flush();
        }
        for (; q < n4; q += nthr) {   // fewer than four float4 left per thread
            const float4 a = __ldcs(p4 + q), b = __ldcs(m4 + q);
            acc.add(a.x, b.x); acc.add(a.y, b.y); acc.add(a.z, b.z); acc.add(a.w, b.w);
        }
        acc.flush();
        done = n4 * 4;
    }
    {
        int n = 0;
        for (size_t idx = done + tid; idx < total; idx += nthr) {
            acc.add(ip[idx], im[idx]);
            if (++n == 32) { acc.flush(); n = 0; }
        }
        acc.flush();
    }
    // block reduction, one warp per quantity over the 256 threads' values in
    // shared memory: a shuffle reduction of all six in every warp kept the
    // FP64 pipe busy longer than the loads took
    bsum[0][threadIdx.x] = acc.sum[0]; bsum[1][threadIdx.x] = acc.sum[1];
    bext[0][threadIdx.x] = acc.mn[0]; bext[1][threadIdx.x] = acc.mn[1];
    bext[2][threadIdx.x] = acc.mx[0]; bext[3][threadIdx.x] = acc.mx[1];
    __syncthreads();
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    double *m = mon + (size_t)blockIdx.x * NM;
    if (q < 2) {
        double t = bsum[q][lane];
#pragma unroll
        for (int r = 1; r < 8; ++r) t += bsum[q][lane + 32 * r];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) m[q] = t * vol;
    } else if (q < 6) {
        const bool lo = q < 4;
        T t = bext[q - 2][lane];
        for (int r = 1; r < 8; ++r) {
            const T x = bext[q - 2][lane + 32 * r];
            t = (lo ? x < t : x > t) ? x : t;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const T x = __shfl_down_sync(0xffffffffu, t, o);
            t = (lo ? x < t : x > t) ? x : t;
        }
        if (lane == 0) m[q] = (double)t;
    }
}

int launch_monitor(it_ctx *c, cudaStream_t s) {
    const double vol = c->dx * c->dx * c->dx;
    const int cur = c->cur;
    if (c->prec == IT_FP32)
        monitor_kernel<float><<<c->nmon, 256, 0, s>>>((const float *)c->n[cur][0], (const float *)c->n[cur][1],
                                                     c->g.cells(), vol, c->d_mon);
    else
        monitor_kernel<double><<<c->nmon, 256, 0, s>>>((const double *)c->n[cur][0], (const double *)c->n[cur][1],
                                                      c->g.cells(), vol, c->d_mon);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// monitor over caller-given FP32 arrays into nblocks x NM values
int launch_monitor_raw_f32(const float *p, const float *m, size_t cells, double vol, double *mon, int nblocks,
                           cudaStream_t s) {
    monitor_kernel<float><<<nblocks, 256, 0, s>>>(p, m, cells, vol, mon);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// ---------------------------------------------------------------------------
// finalize: fixed-order sums of the per-CTA slots and monitor values
//   out[0..NT) tallies, out[NT..NT+NM) monitor, out[NT+NM..+2) released
// ---------------------------------------------------------------------------
// One warp per quantity: lane l takes entries l, l + 32, ..., then shuffles.
// (A block_sum of all twelve sums took 16 us for 304 slots: sixty FP64
// additions per warp at two lanes per clock and a serial tail; this form
// takes 4.2 us.)
__global__ void __launch_bounds__(480)
finalize_kernel(const double *__restrict__ slots, int nslots, const double *__restrict__ mon,
                int nmon, const double *__restrict__ acc, const int *__restrict__ err, double *__restrict__ out) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w < 9) {            // tallies 0..8 (9 is unused)
        const double t = warp_strided_sum(slots, nslots, w, NT, lane);
        if (lane == 0) out[w] = t;
    } else if (w < 11) {    // in-domain ions
        const double t = warp_strided_sum(mon, nmon, w - 9, NM, lane);
        if (lane == 0) out[NT + w - 9] = t;
    } else {                // extremes
        const int q = w - 9;
        const bool lo = q < 4;
        double t = lo ? INFINITY : -INFINITY;
        for (int b = lane; b < nmon; b += 32) {
            const double x = mon[(size_t)b * NM + q];
            t = lo ? fmin(t, x) : fmax(t, x);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double x = __shfl_down_sync(0xffffffffu, t, o);
            t = lo ? fmin(t, x) : fmax(t, x);
        }
        if (lane == 0) out[NT + q] = t;
    }
    if (threadIdx.x == 0) {
        out[9] = 0.0;
        out[NT + NM + 0] = acc[0];
        out[NT + NM + 1] = acc[1];
        out[NT + NM + 2] = (double)*err;
    }
}

int launch_finalize(it_ctx *c, cudaStream_t s) {
    finalize_kernel<<<1, 480, 0, s>>>(c->d_slots, c->nslots, c->d_mon, c->nmon, c->d_acc, c->d_err, c->d_out);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// ---------------------------------------------------------------------------
// deposition
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long floor_div(long long a, long long n) {
    return (a >= 0) ? a / n : -((-a + n - 1) / n);
}

// A track's window of cells on each axis (+-ceil(6 b/dx) around its cell):
// the first cell (wrapped into the axis when periodic, clipped when
// absorbing) and the number of cells, at most the axis.
struct DepWindow { int x, nx, y, ny; };

// Per track and axis: the fraction of the 1D Gaussian factor
// exp(-u^2/b^2)/(sqrt(pi) b) that falls in each cell, summed over the
// periodic images of the cell inside the window +-ceil(6 b/dx) around the
// centre cell (absorbing faces: only the cell itself, if inside); the x table
// carries the track's ions per cm.  One warp per track and axis walks the
// cells from the window's start, so that a cell edge's error function is
// evaluated once, by the lane that owns it, and the next lane takes it by
// shuffle.  (A block per track and axis with two error functions per cell
// took 74 us for 2000 tracks on 256x256, this takes 28.)  Axes longer than
// DEP_SEG cells are cut into nseg pieces, a warp each: one warp alone wrote
// 500000 cells in 2.2 ms.
constexpr int DEP_SEG = 31 * 32;
__global__ void __launch_bounds__(128)
deposit_tables_kernel(const double *__restrict__ tr, long long nt, int nseg, double dx, int nx, int ny, int periodic,
                      double inv_W, double *__restrict__ wx, double *__restrict__ wy, DepWindow *__restrict__ win) {
    const long long unit = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (unit >= 2 * nt * nseg) return;
    const long long t = unit / (2 * nseg);
    const int rest = (int)(unit - t * (2 * nseg)), axis = rest & 1, seg = (rest >> 1) * DEP_SEG;
    const int n = axis ? ny : nx, end = min(n, seg + DEP_SEG);   // cells [seg, end) of the walk
    const double ctr = tr[t * 4 + axis];
    const double b = tr[t * 4 + 3];
    const double f = axis ? 1.0 : tr[t * 4 + 2] * 1e7 * inv_W;   // ions per cm, on the x table
    const long long w = (long long)ceil(6.0 * b / dx);
    const long long ic = (long long)floor(ctr / dx);
    const long long lo = ic - w, hi = ic + w;
    double *out = axis ? (wy + t * ny) : (wx + t * nx);
    int start, count;   // the window on the axis
    if (periodic) {
        start = (int)(lo - n * floor_div(lo, n));
        count = (int)min((long long)n, 2 * w + 1);
    } else {
        const long long c0 = lo > 0 ? lo : 0, c1 = hi < n - 1 ? hi : n - 1;
        start = c1 >= c0 ? (int)c0 : 0;
        count = c1 >= c0 ? (int)(c1 - c0 + 1) : 0;
    }
    if (lane == 0 && seg == 0) {
        int *o = reinterpret_cast<int *>(win + t) + 2 * axis;
        o[0] = start;
        o[1] = count;
    }
    if (periodic && 2 * w + 1 > n) {   // a cell has several images: sum them, lowest first
        for (int i = seg + lane; i < end; i += 32) {
            double sum = 0.0;
            long long ii = i + n * (-floor_div(-(lo - i), n));   // first image >= lo
            for (; ii <= hi; ii += n)
                sum += 0.5 * (erf(((double)(ii + 1) * dx - ctr) / b) - erf(((double)ii * dx - ctr) / b));
            out[i] = f * sum;
        }
        return;
    }
    // cell m of the walk is cell (start + m) mod n; its unwrapped index is
    // first + m, and 31 cells a round share 32 edges
    const long long first = periodic ? lo : start;
    for (int m0 = seg; m0 < end; m0 += 31) {
        const int m = m0 + lane;
        double e = 0.0;
        if (m0 < count) e = m <= count ? erf(((double)(first + m) * dx - ctr) / b) : 0.0;
        const double up = __shfl_down_sync(0xffffffffu, e, 1);
        if (lane < 31 && m < n) {
            int i = start + m;
            if (i >= n) i -= n;
            out[i] = m < count ? f * (0.5 * (up - e)) : 0.0;
        }
    }
}

// Does a window reach the cells [t0, t0 + tn) of an axis of n cells?
__device__ __forceinline__ bool window_hits(int start, int count, int t0, int tn, int n, bool periodic) {
    if (!periodic) return start < t0 + tn && start + count > t0;
    int d = t0 - start;
    if (d < 0) d += n;
    return d < count || d + tn - 1 >= n;
}

constexpr int DEP_TILE = 8;       // 8 x 8 cells per CTA
constexpr int DEP_LIST = 512;     // tracks gathered per pass
constexpr size_t DEP_BLOCKS = 152 * 32 * 4;   // four rounds of resident blocks; fixed, so the sums are deterministic

// plane[j][i] = sum_t N0_t wx[t][i] wy[t][j] / dx^2, tracks in index order.
// Each CTA first lists (in index order) the tracks whose window reaches its
// tile, then every cell sums over that list; tracks that miss the tile only
// contribute zeros, so the per-cell sum is the same as over all tracks.
// part[blockIdx] receives the sum of the plane over the block's tiles (FP64);
// a block takes tiles blockIdx.x, blockIdx.x + gridDim.x, ... (one, up to
// DEP_BLOCKS tiles; with a block each a single track on 4096x4096 took 770 us,
// 192 so, most of it for 262144 FP64 reductions and the sum of the parts).
// Bound by the chain of additions per cell and by the scan; small tiles keep the lists
// short and give a 48x48 section 36 CTAs (16x16 tiles with 64-bit window
// arithmetic in every scan: 93 us on 256x256 with 2000 tracks and 120 us on
// 48x48 with up to 500; this: 23 and 30).
__global__ void __launch_bounds__(DEP_TILE *DEP_TILE)
deposit_plane_kernel(const DepWindow *__restrict__ win, const double *__restrict__ wx, const double *__restrict__ wy,
                     long long nt, int nx, int ny, unsigned ntiles, int periodic, double inv_dx2,
                     double *__restrict__ plane, double *__restrict__ part) {
    constexpr int NTH = DEP_TILE * DEP_TILE, NWARP = NTH / 32;
    __shared__ int list[DEP_LIST];
    __shared__ int wcount[NWARP];
    __shared__ double stage[16][16];   // [track][8 column weights, 8 row weights]
    __shared__ double red[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned ntx = (unsigned)(nx + DEP_TILE - 1) / DEP_TILE;   // tiles in raster order
    double all = 0.0;   // this thread's cells of all the block's tiles
    for (unsigned tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int i0 = (int)(tile % ntx) * DEP_TILE, j0 = (int)(tile / ntx) * DEP_TILE;
        const int tnx = min(DEP_TILE, nx - i0), tny = min(DEP_TILE, ny - j0);
        const bool inside = (tid % DEP_TILE) < tnx && (tid / DEP_TILE) < tny;
        const int i = i0 + (tid % DEP_TILE), j = j0 + (tid / DEP_TILE);
        double sum = 0.0;
        for (long long base = 0; base < nt;) {
            // gather up to DEP_LIST candidates in index order, NTH tracks per round
            int n = 0;
            long long t0 = base;
            for (; t0 < nt && n + NTH <= DEP_LIST; t0 += NTH) {
                const long long t = t0 + tid;
                bool hit = false;
                if (t < nt) {
                    const DepWindow w = win[t];
                    hit = window_hits(w.x, w.nx, i0, tnx, nx, periodic != 0) &&
                          window_hits(w.y, w.ny, j0, tny, ny, periodic != 0);
                }
                const unsigned bal = __ballot_sync(0xffffffffu, hit);
                if (lane == 0) wcount[warp] = __popc(bal);
                __syncthreads();
                int before = 0, total = 0;
#pragma unroll
                for (int q = 0; q < NWARP; ++q) {
                    if (q < warp) before += wcount[q];
                    total += wcount[q];
                }
                if (hit) list[n + before + __popc(bal & ((1u << lane) - 1u))] = (int)t;
                n += total;
                __syncthreads();
            }
            // the listed tracks' weights on the tile's columns and rows, 16 tracks
            // at a time through shared memory (the next 16 are loaded while these
            // are added, in order)
            double r[4];
            auto fetch = [&](int q0) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int idx = tid + NTH * e, q = q0 + (idx >> 4), w = idx & 15;
                    r[e] = 0.0;
                    if (q < n) {
                        const long long t = list[q];
                        r[e] = w < DEP_TILE ? wx[t * nx + min(i0 + w, nx - 1)] : wy[t * ny + min(j0 + w - DEP_TILE, ny - 1)];
                    }
                }
            };
            fetch(0);
            for (int q0 = 0; q0 < n; q0 += 16) {
                __syncthreads();
#pragma unroll
                for (int e = 0; e < 4; ++e) stage[(tid + NTH * e) >> 4][(tid + NTH * e) & 15] = r[e];
                __syncthreads();
                if (q0 + 16 < n) fetch(q0 + 16);
#pragma unroll
                for (int t = 0; t < 16; ++t) sum = fma(stage[t][tid % DEP_TILE], stage[t][DEP_TILE + tid / DEP_TILE], sum);
            }
            base = t0;
            __syncthreads();
        }
        const double v = sum * inv_dx2;
        if (inside) {
            plane[(size_t)j * nx + i] = v;
            all += v;
        }
    }
    double r[1] = {all};
    block_sum<1>(r, red);
    if (tid == 0) part[blockIdx.x] = r[0];
}

// n += plane on every z plane.  Thread = V adjacent columns (float4 when the
// state is FP32 and nx % 4 == 0) over a chunk of DEP_KCHUNK planes
// (blockIdx.y); columns the deposit did not reach are skipped.  FP32 states
// add the plane value rounded to FP32 (n + float(plane), one FP32 addition:
// FP64 arithmetic is slow on this GPU and the two roundings stay within an
// ulp of the exact sum); FP64 states add it exactly in FP64.
constexpr int DEP_KCHUNK = 8;
template <typename T, int V>
__global__ void __launch_bounds__(256)
deposit_apply_kernel(T *__restrict__ p, T *__restrict__ m, const double *__restrict__ plane, size_t plane_n,
                     int nz) {
    const size_t c0 = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * V;
    if (c0 >= plane_n) return;
    double a[V];
    bool any = false;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        a[v] = plane[c0 + v];
        any |= a[v] != 0.0;
    }
    if (!any) return;   // x + 0 == x: nothing to write
    const int k0 = blockIdx.y * DEP_KCHUNK, k1 = min(nz, k0 + DEP_KCHUNK);
    if constexpr (V == 4) {
        const float4 af = make_float4(__double2float_rn(a[0]), __double2float_rn(a[1]), __double2float_rn(a[2]),
                                      __double2float_rn(a[3]));
        float4 *p4 = reinterpret_cast<float4 *>(p), *m4 = reinterpret_cast<float4 *>(m);
        for (int k = k0; k < k1; ++k) {
            const size_t i4 = ((size_t)k * plane_n + c0) / 4;
            float4 x = p4[i4], y = m4[i4];
            x.x = __fadd_rn(x.x, af.x); x.y = __fadd_rn(x.y, af.y); x.z = __fadd_rn(x.z, af.z); x.w = __fadd_rn(x.w, af.w);
            y.x = __fadd_rn(y.x, af.x); y.y = __fadd_rn(y.y, af.y); y.z = __fadd_rn(y.z, af.z); y.w = __fadd_rn(y.w, af.w);
            p4[i4] = x;
            m4[i4] = y;
        }
    } else if constexpr (sizeof(T) == 4) {
        const float af = __double2float_rn(a[0]);
        for (int k = k0; k < k1; ++k) {
            const size_t idx = (size_t)k * plane_n + c0;
            p[idx] = __fadd_rn(p[idx], af);
            m[idx] = __fadd_rn(m[idx], af);
        }
    } else {
        for (int k = k0; k < k1; ++k) {
            const size_t idx = (size_t)k * plane_n + c0;
            p[idx] += a[0];
            m[idx] += a[0];
        }
    }
}

// released += sum(tile sums) * dx^2 * (nz dx) for both species, fixed order
__global__ void __launch_bounds__(256)
deposit_released_kernel(const double *__restrict__ part, size_t n, double factor, double *__restrict__ acc) {
    __shared__ double red[32];
    double v[1] = {0.0};
    for (size_t q = threadIdx.x; q < n; q += blockDim.x) v[0] += part[q];
    block_sum<1>(v, red);
    if (threadIdx.x == 0) {
        acc[0] += v[0] * factor;
        acc[1] += v[0] * factor;
    }
}

int launch_deposit(it_ctx *c, int64_t n, cudaStream_t s) {
    if (n <= 0) return IT_OK;
    const int nx = c->g.nx, ny = c->g.ny;
    const bool periodic = c->p.lateral_bc == IT_PERIODIC;
    DepWindow *win = reinterpret_cast<DepWindow *>(c->d_tracks + 4 * n);   // after the track records
    const int nseg = (std::max(nx, ny) + DEP_SEG - 1) / DEP_SEG;
    deposit_tables_kernel<<<(unsigned)((2 * n * nseg + 3) / 4), 128, 0, s>>>(c->d_tracks, n, nseg, c->dx, nx, ny, periodic,
                                                                            1.0 / c->p.W_eV, c->d_wx, c->d_wy, win);
    IT_CK(cudaGetLastError());
    const long long pn = (long long)nx * ny;
    const size_t ntiles = (size_t)((nx + DEP_TILE - 1) / DEP_TILE) * ((ny + DEP_TILE - 1) / DEP_TILE);
    const size_t nparts = std::min(ntiles, DEP_BLOCKS);
    // the tile sums go after the plane in the same scratch buffer
    double *part = c->d_plane + pn;
    deposit_plane_kernel<<<(unsigned)nparts, DEP_TILE * DEP_TILE, 0, s>>>(
        win, c->d_wx, c->d_wy, n, nx, ny, (unsigned)ntiles, periodic ? 1 : 0, 1.0 / (c->dx * c->dx), c->d_plane, part);
    IT_CK(cudaGetLastError());
    const unsigned kchunks = (unsigned)((c->g.nz + DEP_KCHUNK - 1) / DEP_KCHUNK);
    if (c->prec == IT_FP32 && nx % 4 == 0)
        deposit_apply_kernel<float, 4><<<dim3((unsigned)((pn / 4 + 255) / 256), kchunks), 256, 0, s>>>(
            (float *)c->n[c->cur][0], (float *)c->n[c->cur][1], c->d_plane, (size_t)pn, c->g.nz);
    else if (c->prec == IT_FP32)
        deposit_apply_kernel<float, 1><<<dim3((unsigned)((pn + 255) / 256), kchunks), 256, 0, s>>>(
            (float *)c->n[c->cur][0], (float *)c->n[c->cur][1], c->d_plane, (size_t)pn, c->g.nz);
    else
        deposit_apply_kernel<double, 1><<<dim3((unsigned)((pn + 255) / 256), kchunks), 256, 0, s>>>(
            (double *)c->n[c->cur][0], (double *)c->n[c->cur][1], c->d_plane, (size_t)pn, c->g.nz);
    IT_CK(cudaGetLastError());
    const double factor = c->dx * c->dx * (c->dx * c->g.nz);
    deposit_released_kernel<<<1, 256, 0, s>>>(part, nparts, factor, c->d_acc);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// ---------------------------------------------------------------------------
// tracks at an angle theta to the field (Fig. setup (a))
// ---------------------------------------------------------------------------

// Sum of the cell weights (erf(hi/w) - erf(lo/w))/2 of a profile of width w
// centred at c over the images of cell q in the window [lo_c, hi_c] (cell
// indices, unwrapped): every q + m n inside it when periodic, q itself when not.
__device__ __forceinline__ double image_weights(int q, int n, int lo_c, int hi_c, double c, double w, double dx,
                                                bool periodic) {
    int m0 = 0, m1 = 0;
    if (periodic) {
        // smallest m with q + m n >= lo_c (a ceiling) and largest with
        // q + m n <= hi_c (a floor); C division truncates toward zero
        const int a = lo_c - q, bb = hi_c - q;
        m0 = a >= 0 ? (a + n - 1) / n : -((-a) / n);
        m1 = bb >= 0 ? bb / n : -((-bb + n - 1) / n);
    } else if (q < lo_c || q > hi_c) {
        return 0.0;
    }
    double s = 0.0;
    for (int m = m0; m <= m1; ++m) {
        const double lo = (double)(q + m * n) * dx;
        s += 0.5 * (erf((lo + dx - c) / w) - erf((lo - c) / w));
    }
    return s;
}

// One thread per cell (grid-stride, fixed grid), the tracks in order.  Track
// record [5]: x0, y0, N0 (ions/cm), b, theta.  In the plane of cell centres
// z_k the tilted column's cross-section is the Gaussian of width b/cos(theta)
// in x centred at x0 + (z_k - d/2) tan(theta) and of width b in y:
// (N0/cos) wx wy / dx^2 with the cell weights wx, wy over +-ceil(6 w/dx)
// cells (images summed when periodic).  Within cos(theta) dx / b < 1e-3 of
// parallel to the electrodes the track is one column through the box and wx
// is the cell-centre value dx exp(-u^2/b^2)/(sqrt(pi) b/cos) with
// u = (x - x0) cos - (z_k - d/2) sin: N0/(sqrt(pi) b) exp(-u^2/b^2) wy/dx.
// FP32 states add the FP64 sum rounded once, as the parallel deposit does.
// Each block writes its FP64 sum of the added densities (fixed order).
template <typename T>
__global__ void __launch_bounds__(256)
deposit_angled_kernel(const double *__restrict__ tr, int n, int nx, int ny, int nz, double dx, int periodic,
                      T *__restrict__ p, T *__restrict__ m, double *__restrict__ part) {
    __shared__ double red[32];
    const double zmid = 0.5 * nz * dx;
    const double sqrt_pi = 1.7724538509055160272981674833411;
    const size_t cells = (size_t)nx * ny * nz;
    double bsum[1] = {0.0};
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < cells;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(idx % (size_t)nx);
        const int j = (int)((idx / (size_t)nx) % (size_t)ny);
        const int k = (int)(idx / ((size_t)nx * ny));
        const double zk = (k + 0.5) * dx;
        double v = 0.0;
        for (int t = 0; t < n; ++t) {
            const double x0 = tr[5 * t], y0 = tr[5 * t + 1], N0 = tr[5 * t + 2], b = tr[5 * t + 3];
            const double th = tr[5 * t + 4];
            const int wy = (int)ceil(6.0 * b / dx), jc = (int)floor(y0 / dx);
            const double sy = image_weights(j, ny, jc - wy, jc + wy, y0, b, dx, periodic);
            if (sy == 0.0) continue;
            const double c = cos(th), sn = sin(th);
            if (c * dx / b < 1e-3) {
                const double u = ((i + 0.5) * dx - x0) * c - (zk - zmid) * sn;
                v += N0 / (sqrt_pi * b) * exp(-(u * u) / (b * b)) * sy / dx;
            } else {
                const double xc = x0 + (zk - zmid) * sn / c;
                const int wx = (int)ceil(6.0 * b / (dx * c)), ic = (int)floor(xc / dx);
                const double sx = image_weights(i, nx, ic - wx, ic + wx, xc, b / c, dx, periodic);
                v += (N0 / c) * sx * sy / (dx * dx);
            }
        }
        if (v != 0.0) {
            if constexpr (sizeof(T) == 4) {
                const float vf = __double2float_rn(v);
                p[idx] = __fadd_rn(p[idx], vf);
                m[idx] = __fadd_rn(m[idx], vf);
            } else {
                p[idx] += v;
                m[idx] += v;
            }
            bsum[0] += v;
        }
    }
    block_sum<1>(bsum, red);
    if (threadIdx.x == 0) part[blockIdx.x] = bsum[0];
}

// The same deposit from tables, for the few tracks it is meant for: in every
// plane a tilted column is an x profile times a y profile, so the error
// functions (and, parallel to the electrodes, the exponential) are evaluated
// once per (track, plane, column) and once per (track, row), not once per
// cell and track.  ay[t][j] holds wy; ax[t][k][i] holds wx with the track's
// ions per cm and 1/dx^2, so a cell adds one product per track.
// One warp per row of a table; lane 0 writes the row's sum: rows [0, n) are
// the y rows, row n + t nz + k the x row of track t and plane k.
__global__ void __launch_bounds__(128)
angled_tables_kernel(const double *__restrict__ tr, int n, int nx, int ny, int nz, double dx, int periodic,
                     double *__restrict__ ax, double *__restrict__ ay, double *__restrict__ rowsum) {
    const long long row = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= (long long)n * (nz + 1)) return;
    const double zmid = 0.5 * nz * dx;
    const double sqrt_pi = 1.7724538509055160272981674833411;
    double sum = 0.0;
    if (row < n) {
        const double y0 = tr[5 * row + 1], b = tr[5 * row + 3];
        const int w = (int)ceil(6.0 * b / dx), jc = (int)floor(y0 / dx);
        for (int j = lane; j < ny; j += 32) {
            const double v = image_weights(j, ny, jc - w, jc + w, y0, b, dx, periodic);
            ay[row * ny + j] = v;
            sum += v;
        }
    } else {
        const long long q = row - n;
        const int t = (int)(q / nz), k = (int)(q - (long long)t * nz);
        const double x0 = tr[5 * t], N0 = tr[5 * t + 2], b = tr[5 * t + 3], th = tr[5 * t + 4];
        const double zk = (k + 0.5) * dx;
        double *out = ax + q * nx;
        const double c = cos(th), sn = sin(th);
        if (c * dx / b < 1e-3) {
            for (int i = lane; i < nx; i += 32) {
                const double u = ((i + 0.5) * dx - x0) * c - (zk - zmid) * sn;
                const double v = N0 / (sqrt_pi * b) * exp(-(u * u) / (b * b)) / dx;
                out[i] = v;
                sum += v;
            }
        } else {
            const double xc = x0 + (zk - zmid) * sn / c;
            const int w = (int)ceil(6.0 * b / (dx * c)), ic = (int)floor(xc / dx);
            const double f = N0 / c / (dx * dx);
            for (int i = lane; i < nx; i += 32) {
                const double v = f * image_weights(i, nx, ic - w, ic + w, xc, b / c, dx, periodic);
                out[i] = v;
                sum += v;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    if (lane == 0) rowsum[row] = sum;
}

// n += sum over the tracks of ax[t][k][i] ay[t][j].  Thread = V adjacent
// cells of a row (float4 when the state is FP32 and nx % 4 == 0); cells no
// track reaches are neither read nor written.  FP32 states add the FP64 sum
// rounded once, as the other deposits do.
template <typename T, int V, typename Idx>
__global__ void __launch_bounds__(256)
angled_apply_kernel(const double *__restrict__ ax, const double *__restrict__ ay, int n, int nx, int ny, int nz,
                    T *__restrict__ p, T *__restrict__ m) {
    const Idx nxv = (Idx)(nx / V);
    const Idx total = nxv * (Idx)ny * (Idx)nz;
    for (Idx e = (Idx)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (Idx)gridDim.x * blockDim.x) {
        const Idx r = e / nxv;
        const int i = (int)(e - r * nxv) * V, k = (int)(r / (Idx)ny), j = (int)(r - (Idx)k * (Idx)ny);
        double v[V] = {};
        bool any = false;
        for (int t = 0; t < n; ++t) {
            const double y = ay[(long long)t * ny + j];
            if (y == 0.0) continue;
            const double *x = ax + ((long long)t * nz + k) * nx + i;
#pragma unroll
            for (int q = 0; q < V; ++q) {
                const double xv = x[q];
                v[q] = fma(xv, y, v[q]);
                any |= xv != 0.0;
            }
        }
        if (!any) continue;
        const size_t idx = (size_t)r * nx + i;
        if constexpr (V == 4) {
            float4 a = *reinterpret_cast<float4 *>(p + idx), b = *reinterpret_cast<float4 *>(m + idx);
            const float4 f = make_float4(__double2float_rn(v[0]), __double2float_rn(v[1]), __double2float_rn(v[2]),
                                         __double2float_rn(v[3]));
            a.x = __fadd_rn(a.x, f.x); a.y = __fadd_rn(a.y, f.y); a.z = __fadd_rn(a.z, f.z); a.w = __fadd_rn(a.w, f.w);
            b.x = __fadd_rn(b.x, f.x); b.y = __fadd_rn(b.y, f.y); b.z = __fadd_rn(b.z, f.z); b.w = __fadd_rn(b.w, f.w);
            *reinterpret_cast<float4 *>(p + idx) = a;
            *reinterpret_cast<float4 *>(m + idx) = b;
        } else if constexpr (sizeof(T) == 4) {
            const float f = __double2float_rn(v[0]);
            p[idx] = __fadd_rn(p[idx], f);
            m[idx] = __fadd_rn(m[idx], f);
        } else {
            p[idx] += v[0];
            m[idx] += v[0];
        }
    }
}

// released += sum over tracks and planes of (x row sum) (y row sum) * vol
__global__ void __launch_bounds__(256)
angled_released_kernel(const double *__restrict__ rowsum, int n, int nz, double vol, double *__restrict__ acc) {
    __shared__ double red[32];
    double v[1] = {0.0};
    const long long rows = (long long)n * nz;
    for (long long q = threadIdx.x; q < rows; q += blockDim.x) v[0] = fma(rowsum[n + q], rowsum[q / nz], v[0]);
    block_sum<1>(v, red);
    if (threadIdx.x == 0) {
        acc[0] += v[0] * vol;
        acc[1] += v[0] * vol;
    }
}

// Doubles of scratch the tables of n tracks take, 0 where the kernel without
// tables is used: the x tables hold nz nx doubles per track, so many tracks
// on a large section would outgrow the section's own state.  Up to 256 MB
// (26 tracks on 200x200x800) the tables win by far: one iron track there
// takes 0.25 ms against 19.5 (0.19 of it adds 32M cells, bound by the FP64
// product and conversion per cell).
int64_t angled_table_doubles(const it_ctx *c, int64_t n) {
    const double need = (double)n * ((double)c->g.nz * c->g.nx + c->g.ny + c->g.nz + 1);
    if (need * sizeof(double) > 256.0 * 1024 * 1024) return 0;
    return (int64_t)need;
}

int launch_deposit_angled(it_ctx *c, const double *d_tr, int64_t n, double *d_part, int nblocks, double *d_tab,
                          cudaStream_t s) {
    if (n <= 0) return IT_OK;
    const int nx = c->g.nx, ny = c->g.ny, nz = c->g.nz;
    const int per = c->p.lateral_bc == IT_PERIODIC ? 1 : 0;
    const double vol = c->dx * c->dx * c->dx;
    if (d_tab) {
        double *ax = d_tab, *ay = ax + n * nz * (int64_t)nx, *rowsum = ay + n * ny;
        const long long rows = n * (nz + 1);
        angled_tables_kernel<<<(unsigned)((rows + 3) / 4), 128, 0, s>>>(d_tr, (int)n, nx, ny, nz, c->dx, per, ax, ay,
                                                                       rowsum);
        IT_CK(cudaGetLastError());
        const int cur = c->cur;
        const size_t cells = c->g.cells();
        const bool small = cells <= 0xf0000000ull;
        const bool v4 = c->prec == IT_FP32 && nx % 4 == 0;
        const size_t items = v4 ? cells / 4 : cells;
        // a few rounds per thread on large grids
        const unsigned grid = (unsigned)std::min<size_t>((items + 255) / 256, 152 * 64);
        auto go = [&](auto *k, auto *pp, auto *mm) { k<<<grid, 256, 0, s>>>(ax, ay, (int)n, nx, ny, nz, pp, mm); };
        float *pf = (float *)c->n[cur][0], *mf = (float *)c->n[cur][1];
        double *pd = (double *)c->n[cur][0], *md = (double *)c->n[cur][1];
        if (v4) small ? go(angled_apply_kernel<float, 4, uint32_t>, pf, mf) : go(angled_apply_kernel<float, 4, uint64_t>, pf, mf);
        else if (c->prec == IT_FP32) small ? go(angled_apply_kernel<float, 1, uint32_t>, pf, mf) : go(angled_apply_kernel<float, 1, uint64_t>, pf, mf);
        else small ? go(angled_apply_kernel<double, 1, uint32_t>, pd, md) : go(angled_apply_kernel<double, 1, uint64_t>, pd, md);
        IT_CK(cudaGetLastError());
        angled_released_kernel<<<1, 256, 0, s>>>(rowsum, (int)n, nz, vol, c->d_acc);
        IT_CK(cudaGetLastError());
        return IT_OK;
    }
    if (c->prec == IT_FP32)
        deposit_angled_kernel<float><<<nblocks, 256, 0, s>>>(d_tr, (int)n, nx, ny, nz, c->dx, per,
                                                             (float *)c->n[c->cur][0], (float *)c->n[c->cur][1],
                                                             d_part);
    else
        deposit_angled_kernel<double><<<nblocks, 256, 0, s>>>(d_tr, (int)n, nx, ny, nz, c->dx, per,
                                                              (double *)c->n[c->cur][0],
                                                              (double *)c->n[c->cur][1], d_part);
    IT_CK(cudaGetLastError());
    deposit_released_kernel<<<1, 256, 0, s>>>(d_part, (size_t)nblocks, vol, c->d_acc);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

int launch_zero(void *p, size_t bytes, cudaStream_t s) {
    IT_CK(cudaMemsetAsync(p, 0, bytes, s));
    return IT_OK;
}

}  // namespace itk
