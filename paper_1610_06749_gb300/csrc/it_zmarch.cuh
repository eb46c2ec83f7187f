// it_zmarch.cuh -- the bandwidth-bound step kernel for FP32 densities.
//
// One explicit step of the Appendix scheme for both species (Lax-Wendroff
// drift along z, 3-point diffusion on each axis, -alpha n+ n- from the old
// level; Eq. theEquation without space charge) with the electrode/lateral
// collection and recombination tallies fused in.
//
// Layout and data movement:
//   * a CTA owns TY full-width rows (y0 .. y0+TY-1) of one y-tile and marches
//     up or down a chunk of z planes [z0, z1);
//   * every plane it needs (z0-1 .. z1) arrives in a shared-memory slot by TMA
//     (cp.async.bulk.tensor, 3-D tiles of n+ and n-): TY main rows plus one
//     halo row above and below, wrapped when the lateral faces are periodic.
//     Rows and planes outside the tensor (the absorbing faces' ghost rows, the
//     electrode ghost planes z = -1 and z = nz) are filled with zeros by TMA,
//     which is exactly the boundary condition n = 0;
//   * an S-deep ring of slots keeps S-2 planes in flight while one plane is
//     computed; a producer warp refills a slot when its readers have left it;
//   * each thread owns float4 x-segments and keeps the last plane's and this
//     plane's values in registers; x and y neighbours and the next plane come
//     from shared memory;
//     the update runs on paired FP32 instructions (two cells per instruction);
//   * results are stored with coalesced 16-byte stores; per-thread FP32
//     partial sums (at most 32 planes; with their rounding errors on EXACT
//     instances) are reduced per warp in FP64 and per CTA into the CTA's own
//     tally slot (deterministic).
// Every mbarrier wait is bounded: a ring wait that runs out (after
// zc.wait_cycles SM cycles, 2^32 by default) raises the device error flag,
// and the CTA waits, with the full 2^32-cycle bound, for the copies it has
// issued and returns.  A test hook (zc.withhold) leaves the first ring load
// unissued, so that every warp's first wait runs out without any fault.
#pragma once

#include <algorithm>

#include "it_device.cuh"
#include "it_internal.cuh"
#include "it_tma.cuh"

namespace itk {

struct ZmMaps {
    CUtensorMap main[2];   // n+, n- of the input set
    CUtensorMap halo[2];
};

constexpr int ZM_MAX_IPT = 4;                    // float4 items per thread
constexpr int ZM_MAX_SEG = 8;                    // segments of a CTA kept in shared memory

// Persistent step kernel: NW warps that compute and, where PROD, one that
// loads.
//   The planes a CTA needs stream through an S-deep ring of shared-memory
//   slots by TMA.  full[slot] completes when a plane's bytes have landed.
//   PROD: one thread of an extra warp walks the CTA's planes, waits on
//   empty[slot] (one arrival per computing warp) and loads the next plane.
//   Otherwise every warp, after its reads of a slot, adds one to the slot's
//   release counter, and the warp whose release completes the count refills
//   the slot.  That refill is done by the warp the others wait for and adds
//   about 1.2 us to every plane: 256x256x400, 8 rows, 2 CTAs per SM, ring of
//   4: 73.6 us with the producer, 77 without (the loads and stores alone,
//   with nothing computed, take 70 to 80); 512x512x256, 8 rows, 1 CTA per SM:
//   170 against 195; 200x200x800 absorbing, 8 rows, 2 CTAs: 88 against 95.
//   The ninth warp costs registers, though: 96 per thread instead of 128,
//   which spills with space charge (384x320x128: 56.3 us with the producer,
//   53.1 without), with more than two float4 per thread (32 rows of
//   256x256x400: 142 against 83) and with two that are no pair beside
//   absorbing faces, so those keep the refill by the last reader.
//   Every warp marches along z, one plane per iteration, with no block-wide
//   barrier inside the march.  DOWN: the CTA walks its planes downwards.
//   Steps alternate between up and down, so that a step first reads the
//   planes which the step before it wrote last and which are still in L2
//   (256x256x400: 73.6 to 69.8 us); the update of a cell is the same
//   operations either way.
//   PAIR: a thread's two float4 lie one above the other, so each is the
//   other's y neighbour: 4 shared-memory reads of 16 bytes per pair and
//   species instead of 6.
//   EXACT: the per-thread sums carry the rounding error of each addition
//   (CompSum), so the tallies are as close as FP64 sums of the FP32 terms.
//   For rows of more than 256 cells that are no multiple of 256, whose tallies
//   the simple kernel sums that closely too.  It costs up to 6 % of a step
//   (384x320x128: 49.7 us with it, 48.8 with plain sums; absorbing faces 55.6
//   and 55.2, 320x256x200 61.6 and 58.3, 640x384x100 78.9 and 76.0), so the
//   other widths keep the plain sums they always had (256x256x400 would take
//   72.0 us instead of 71.2).
//   The FP64 tallies live in shared memory (each warp's lane 0 adds to its
//   own row), so the registers hold only the marching planes and offsets.
__host__ __device__ constexpr bool zm_prod(bool periodic, int ipt, bool sc, bool pair) {
    return !sc && (ipt == 1 || (ipt == 2 && (periodic || pair)));
}

// one thread's sum of a tally over up to 32 planes
template <bool EXACT>
struct RingSum {   // plain FP32
    float v = 0.f;
    __device__ __forceinline__ void add(float2 a, float2 b) { v += (a.x + a.y) + (b.x + b.y); }
    __device__ __forceinline__ double value() const { return (double)v; }
};
template <>
struct RingSum<true> {
    CompSum2 c;
    __device__ __forceinline__ void add(float2 a, float2 b) { c.term(a); c.term(b); }
    __device__ __forceinline__ double value() const { return c.total().value(); }
};

template <bool PERIODIC, int IPT, int NW, bool SC, bool PAIR, bool DOWN, bool EXACT>
__global__ void __launch_bounds__(NW * 32 + (zm_prod(PERIODIC, IPT, SC, PAIR) ? 32 : 0), (NW <= 8 ? 2 : 1))
step_zmarch_kernel(const __grid_constant__ ZmMaps maps, const float *__restrict__ inp,
                   const float *__restrict__ inm, float *__restrict__ outp, float *__restrict__ outm,
                   int nx, int ny, int nz, const ZmConf zc, const Coef<float> cf, double *__restrict__ slots,
                   int *__restrict__ err) {
    constexpr int NT_ = NW * 32;
    constexpr bool PROD = zm_prod(PERIODIC, IPT, SC, PAIR);
    extern __shared__ __align__(128) unsigned char zm_smem_raw[];
    // TMA destinations need 128-byte alignment: round the base up explicitly
    unsigned char *smem_base = zm_smem_raw + ((128u - (smem_u32(zm_smem_raw) & 127u)) & 127u);
    float *ring = reinterpret_cast<float *>(smem_base);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem_base + (size_t)zc.S * zc.slot * sizeof(float));
    uint64_t *empty = full + zc.S;                                 // PROD: the slot's readers are done with it
    uint32_t *rel = reinterpret_cast<uint32_t *>(full + zc.S);     // else: release counters
    uint32_t *fills = rel + zc.S;                                  // loads issued per slot
    // per-warp FP64 tallies (tally q of warp w at w*WQ+q): 7 tallies, 9 with
    // space charge; a power-of-two row keeps the index a shift
    constexpr int WQ = SC ? 16 : 8, NQ = SC ? 9 : 7;
    __shared__ double wacc[NW * WQ];
    __shared__ volatile int abort_flag;
    __shared__ int seg_n0[ZM_MAX_SEG], seg_t[ZM_MAX_SEG], seg_first[ZM_MAX_SEG];   // !PROD

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int ncol4 = nx >> 2;
    const int nitems = ncol4 * zc.TY;
    const int S = zc.S;
    const long long total = (long long)zc.ntile * nz;
    const long long g0 = total * blockIdx.x / gridDim.x;
    const long long g1 = total * (blockIdx.x + 1) / gridDim.x;

    // load plane p of tile t into a slot (one thread)
    auto load = [&](int t, int p, int slot) {
        const int y0 = t * zc.TY;
        // halo rows: wrapped when periodic; rows -1 and ny otherwise, which
        // lie outside the tensor and arrive as zeros (absorbing faces hold
        // n = 0); planes -1 and nz arrive as zeros the same way
        const int ytop = PERIODIC ? (y0 > 0 ? y0 - 1 : ny - 1) : y0 - 1;
        const int ybot = PERIODIC ? (y0 + zc.TY < ny ? y0 + zc.TY : 0) : y0 + zc.TY;
        const uint32_t tx = 2u * (uint32_t)(zc.TY + 2) * zc.bx * 4u;
        float *base = ring + (size_t)slot * zc.slot;
        uint64_t *bar = &full[slot];
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, tx);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            float *blk = base + (size_t)s * zc.blk;
            if (zc.xs > 1) {
                // whole rows of a wide grid in one box
                tma_load4(blk + zc.reg_main, &maps.main[s], bar, 0, 0, y0, p);
                tma_load4(blk + zc.reg_top, &maps.halo[s], bar, 0, 0, ytop, p);
                tma_load4(blk + zc.reg_bot, &maps.halo[s], bar, 0, 0, ybot, p);
            } else {
                tma_load3(blk + zc.reg_main, &maps.main[s], bar, 0, y0, p);
                tma_load3(blk + zc.reg_top, &maps.halo[s], bar, 0, ytop, p);
                tma_load3(blk + zc.reg_bot, &maps.halo[s], bar, 0, ybot, p);
            }
        }
    };

    // without a producer: planes this CTA loads (every segment [za, zb) loads
    // zb - za + 2).  The first ZM_MAX_SEG segments are also kept in shared
    // memory (first sequence number, tile, lowest plane, count), so that a
    // refill finds its plane without the 64-bit divisions of the walk: a
    // refill lies on the critical path, since the warp that issues it is the
    // last one done with the slot
    int nload = 0;
    int nseg = 0;
    if constexpr (!PROD) {
        Segs sg{g0, g1, nz, 0, 0, 0};
        while (sg.next()) {
            if (tid == 0 && nseg < ZM_MAX_SEG) {
                seg_n0[nseg] = nload;
                seg_t[nseg] = sg.t;
                seg_first[nseg] = DOWN ? sg.zb : sg.za - 1;
            }
            ++nseg;
            nload += sg.zb - sg.za + 2;
        }
    }
    // load plane n of the sequence into its slot (one thread)
    auto issue = [&](int n) {
        if (n >= nload) return;
        int t = 0, p = 0;
        if (nseg <= ZM_MAX_SEG) {
            int i = 0;
            while (i + 1 < nseg && n >= seg_n0[i + 1]) ++i;
            t = seg_t[i];
            p = DOWN ? seg_first[i] - (n - seg_n0[i]) : seg_first[i] + (n - seg_n0[i]);
        } else {
            Segs sg{g0, g1, nz, 0, 0, 0};
            int m = n;   // loads of the segments from sg on
            while (sg.next() && m >= sg.zb - sg.za + 2) m -= sg.zb - sg.za + 2;
            t = sg.t;
            p = DOWN ? sg.zb - m : sg.za - 1 + m;
        }
        const int slot = n % S;
        load(t, p, slot);
        fills[slot] += 1;
    };

    if (tid == 0) {
        for (int q = 0; q < S; ++q) {
            mbar_init(&full[q], 1);
            if (PROD) mbar_init(&empty[q], NW);
            if (!PROD) rel[q] = fills[q] = 0;
        }
        for (int q = 0; q < NW * WQ; ++q) wacc[q] = 0.0;
        abort_flag = 0;
        fence_mbar_init();
        if constexpr (!PROD)
            for (int n = zc.withhold ? 1 : 0; n < S && n < nload; ++n) issue(n);
    }
    __syncthreads();

    if constexpr (PROD)
        if (warp == NW) {
            if (lane == 0) {
                RingPos pos{0, 0u};
                int n = 0;
                Segs sg{g0, g1, nz, 0, 0, 0};
                bool stop = false;
                while (!stop && sg.next())
                    for (int q = sg.za - 1; q <= sg.zb; ++q, ++n) {
                        if (n >= S) {
                            // the slot's readers (bounded by zc.wait_cycles)
                            const uint32_t par = pos.phase ^ 1u;
                            if (!mbar_try_wait(&empty[pos.slot], par)) {
                                const long long t0 = clock64();
                                while (!mbar_try_wait(&empty[pos.slot], par))
                                    if (abort_flag || clock64() - t0 > zc.wait_cycles) {
                                        stop = true;
                                        break;
                                    }
                            }
                            if (stop || abort_flag) {
                                stop = true;
                                abort_flag = 1;
                                break;
                            }
                        }
                        if (!(zc.withhold && n == 0)) load(sg.t, DOWN ? sg.za - 1 + sg.zb - q : q, pos.slot);
                        pos.advance(S);
                    }
                if (stop) atomicExch(err, 1);
                // no load may be in flight when the CTA exits: wait (bounded)
                // for the last load issued into each slot
                RingPos d{0, 0u};
                for (int q = 0; q < n; ++q) {
                    if (q + S >= n && !(zc.withhold && q == 0)) (void)mbar_wait_bounded(&full[d.slot], d.phase);
                    d.advance(S);
                }
            }
            __syncwarp();
            __syncthreads();   // the computing warps' last barrier
            return;
        }

    // warp-uniform: reduce one partial per lane in FP64 (fixed shuffle order)
    // and add it to the warp's tally q
    auto flush = [&](int q, double v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) wacc[warp * WQ + q] += v;
    };

    // per-item offsets inside a species block (species 1: + nbx*blk); x
    // neighbours are read from shared memory at wrapped offsets (periodic) or
    // replaced by zero at an absorbing row end
    int o_c[IPT], o_u[IPT], o_d[IPT], o_l[IPT], o_r[IPT], ty_[IPT], c4_[IPT];
    bool valid[IPT];
#pragma unroll
    for (int it = 0; it < IPT; ++it) {
        // items in raster order; as pairs: two vertically adjacent rows
        const int q = tid + (PAIR ? it / 2 : it) * NT_;
        const int nq = PAIR ? nitems / 2 : nitems;
        valid[it] = q < nq;
        const int qe = valid[it] ? q : nq - 1;
        const int ty = PAIR ? 2 * (qe / ncol4) + (it & 1) : qe / ncol4, c4 = qe - (qe / ncol4) * ncol4;
        ty_[it] = ty;
        c4_[it] = c4;
        const int x0 = 4 * c4;
        const int xb = x0 / zc.bx, xi = x0 - xb * zc.bx;
        const int bofs = xb * zc.blk;
        o_c[it] = bofs + zc.reg_main + ty * zc.bx + xi;
        o_u[it] = bofs + (ty == 0 ? zc.reg_top : zc.reg_main + (ty - 1) * zc.bx) + xi;
        o_d[it] = bofs + (ty == zc.TY - 1 ? zc.reg_bot : zc.reg_main + (ty + 1) * zc.bx) + xi;
        const int xl = c4 == 0 ? nx - 1 : x0 - 1;
        const int xr = c4 == ncol4 - 1 ? 0 : x0 + 4;
        o_l[it] = (xl / zc.bx) * zc.blk + zc.reg_main + ty * zc.bx + (xl % zc.bx);
        o_r[it] = (xr / zc.bx) * zc.blk + zc.reg_main + ty * zc.bx + (xr % zc.bx);
    }
    const int sp_ofs = zc.nbx * zc.blk;
    const uint32_t plane = (uint32_t)nx * (uint32_t)ny;
    RingPos pos{0, 0u};
    int nrel = 0;            // planes of the sequence this warp has released
    bool failed = false;

    // Wait (bounded by zc.wait_cycles) for the plane at ring position u.  A
    // lost wait marks the whole warp failed (shuffles stay convergent) and
    // raises the CTA's abort flag, after which no warp waits again.
    auto wait_full = [&](const RingPos &u) {
        if (failed) return;
        bool ok = mbar_try_wait(&full[u.slot], u.phase);
        if (__all_sync(0xffffffffu, ok)) return;
        const long long t0 = clock64();
        for (;;) {
            ok = ok || mbar_try_wait(&full[u.slot], u.phase);
            if (__all_sync(0xffffffffu, ok)) return;
            if (__any_sync(0xffffffffu, abort_flag || clock64() - t0 > zc.wait_cycles)) break;
        }
        failed = true;
        if (lane == 0) abort_flag = 1;
    };
    // After the warp's reads of the slot: hand it back to the producer, or
    // count the release, the last of NW refilling the slot.  A failed warp
    // releases nothing, so no slot is refilled while its previous load may
    // still be in flight.
    auto release = [&](const RingPos &u) {
        __syncwarp();
        if constexpr (PROD) {
            if (lane == 0 && !failed) mbar_arrive(&empty[u.slot]);
        } else {
            if (lane == 0 && !failed) {
                const uint32_t old = atom_add_acq_rel(&rel[u.slot], 1u);
                if (old % NW == NW - 1 && nrel + S < nload && !abort_flag) issue(nrel + S);
            }
            ++nrel;
        }
    };

    if constexpr (EXACT && !PERIODIC) {
        // what leaves through the sides, read again from global memory while
        // the ring fills: summed in the march it holds registers and issue
        // slots that the march needs (384x320x128: 60.3 us, so 55.6)
        CompSum2 lat;   // n+ and n-
        auto cell = [&](uint32_t e) { lat.term(make_float2(__ldg(inp + e), __ldg(inm + e))); };
        Segs sg{g0, g1, nz, 0, 0, 0};
        while (sg.next()) {
            const uint32_t y0 = (uint32_t)(sg.t * zc.TY), n = (uint32_t)(sg.zb - sg.za);
            const uint32_t base = ((uint32_t)sg.za * ny + y0) * nx;   // the tile's first row, plane za
            for (uint32_t q = tid; q < n * zc.TY; q += NT_) {         // row ends
                const uint32_t k = q / zc.TY, e = base + (k * ny + (q - k * zc.TY)) * nx;
                cell(e);
                cell(e + nx - 1);
            }
#pragma unroll
            for (int f = 0; f < 2; ++f) {                             // first and last row of the section
                if (f ? (int)y0 + zc.TY != ny : y0 != 0) continue;
                const uint32_t row = base + (f ? (zc.TY - 1) * nx : 0);
                for (uint32_t q0 = tid; q0 < n * ncol4; q0 += 4 * NT_) {   // four loads of each species in flight
                    float4 P[4], M[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t q = q0 + u * NT_, k = q / ncol4, e = row + k * ny * nx + 4 * (q - k * ncol4);
                        const bool in = q < n * ncol4;
                        P[u] = in ? __ldg(reinterpret_cast<const float4 *>(inp + e)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        M[u] = in ? __ldg(reinterpret_cast<const float4 *>(inm + e)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        lat.term(make_float2(P[u].x, M[u].x));
                        lat.term(make_float2(P[u].y, M[u].y));
                        lat.term(make_float2(P[u].z, M[u].z));
                        lat.term(make_float2(P[u].w, M[u].w));
                    }
                }
            }
        }
        flush(5, CompSum{lat.hi.x, lat.lo.x}.value());
        flush(6, CompSum{lat.hi.y, lat.lo.y}.value());
    }

    Segs seg{g0, g1, nz, 0, 0, 0};
    while (seg.next()) {
        const int za = seg.za, zb = seg.zb;
        const int y0 = seg.t * zc.TY;
        float4 prev[IPT][2], cur[IPT][2];
        uint32_t off[IPT];       // element offset of the item in the current plane (cells < 2^32)
        bool edge_u[IPT], edge_d[IPT];   // rows at an absorbing y face (lateral tally)
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            const int yg = y0 + ty_[it];
            off[it] = ((uint32_t)(DOWN ? zb - 1 : za) * (uint32_t)ny + (uint32_t)yg) * (uint32_t)nx +
                      4u * (uint32_t)c4_[it];
            edge_u[it] = !PERIODIC && yg == 0;
            edge_d[it] = !PERIODIC && yg == ny - 1;
        }
        {
            wait_full(pos);
            const float *sl = ring + (size_t)pos.slot * zc.slot;
#pragma unroll
            for (int it = 0; it < IPT; ++it) {
                prev[it][0] = *reinterpret_cast<const float4 *>(sl + o_c[it]);
                prev[it][1] = *reinterpret_cast<const float4 *>(sl + sp_ofs + o_c[it]);
            }
            release(pos);
            pos.advance(S);
        }
        wait_full(pos);
        RingPos pc = pos;
        pos.advance(S);
        {
            const float *sl = ring + (size_t)pc.slot * zc.slot;
#pragma unroll
            for (int it = 0; it < IPT; ++it) {
                cur[it][0] = *reinterpret_cast<const float4 *>(sl + o_c[it]);
                cur[it][1] = *reinterpret_cast<const float4 *>(sl + sp_ofs + o_c[it]);
            }
        }
        RingSum<EXACT> rsum, ssum[2];
        float lsum0 = 0.f, lsum1 = 0.f;   // !EXACT
        int nacc = 0;
        auto flush_sums = [&]() {
            flush(0, rsum.value());
            rsum = RingSum<EXACT>{};
            if (!PERIODIC && !EXACT) {
                flush(5, (double)lsum0); flush(6, (double)lsum1);
                lsum0 = lsum1 = 0.f;
            }
            if (SC) {
                flush(7, ssum[0].value()); flush(8, ssum[1].value());
                ssum[0] = ssum[1] = RingSum<EXACT>{};
            }
        };
        // not unrolled: an unrolled march (which would save the register
        // rotation of prev/cur) measured slower
        for (int q = za; q < zb; ++q) {
            const int k = DOWN ? za + zb - 1 - q : q;   // the plane computed; prev holds the one walked before it
            const bool electrode = k == 0 || k == nz - 1;
            wait_full(pos);
            const float *sk = ring + (size_t)pc.slot * zc.slot;
            const float *sn = ring + (size_t)pos.slot * zc.slot;
            float an[2] = {0.f, 0.f}, lat[2] = {0.f, 0.f};
            // one item of one species: the update, its store and its tallies
            auto item = [&](int it, int s, float4 n, float4 u, float4 d, float4 zn, float2 rxy, float2 rzw, float2 dxy,
                            float2 dzw) {
                const float *bk = sk + s * sp_ofs;
                float l = bk[o_l[it]];
                float r = bk[o_r[it]];
                if (!PERIODIC) {
                    if (c4_[it] == 0) l = 0.f;
                    if (c4_[it] == ncol4 - 1) r = 0.f;
                }
                float4 v = upd7x4(n, l, r, u, d, DOWN ? zn : prev[it][s], DOWN ? prev[it][s] : zn, rxy, rzw, cf.wx[s],
                                  cf.wzm[s], cf.wzp[s], cf.adt);
                if (SC) {
                    float2 pxy, pzw;
                    v = add_sc4(v, cf.sc[s], n, dxy, dzw, pxy, pzw);
                    if (valid[it]) ssum[s].add(pxy, pzw);
                }
                if (valid[it]) {
                    *reinterpret_cast<float4 *>((s ? outm : outp) + off[it]) = v;
                    if (!EXACT && electrode) an[s] += (n.x + n.y) + (n.z + n.w);
                    if (!PERIODIC && !EXACT) {
                        if (c4_[it] == 0) lat[s] += n.x;
                        if (c4_[it] == ncol4 - 1) lat[s] += n.w;
                        if (edge_u[it]) lat[s] += (n.x + n.y) + (n.z + n.w);
                        if (edge_d[it]) lat[s] += (n.x + n.y) + (n.z + n.w);
                    }
                }
                prev[it][s] = n;
                cur[it][s] = zn;
            };
            auto at = [](const float *q, int o) { return *reinterpret_cast<const float4 *>(q + o); };
#pragma unroll
            for (int it = 0; it < IPT; it += (PAIR ? 2 : 1)) {
                constexpr int W = PAIR ? 2 : 1;   // items at a time
                float2 rxy[W], rzw[W], dxy[W], dzw[W];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const float4 P = cur[it + w][0], M = cur[it + w][1];
                    rxy[w] = __fmul2_rn(make_float2(P.x, P.y), make_float2(M.x, M.y));
                    rzw[w] = __fmul2_rn(make_float2(P.z, P.w), make_float2(M.z, M.w));
                    if (SC) sc_diff4(P, M, dxy[w], dzw[w]);
                }
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const float *bk = sk + s * sp_ofs, *bn = sn + s * sp_ofs;
                    if constexpr (PAIR) {
                        // the two rows are each other's y neighbours
                        const float4 n0 = cur[it][s], n1 = cur[it + 1][s];
                        const float4 u = at(bk, o_u[it]), d = at(bk, o_d[it + 1]);
                        const float4 z0 = at(bn, o_c[it]), z1 = at(bn, o_c[it + 1]);
                        item(it, s, n0, u, n1, z0, rxy[0], rzw[0], dxy[0], dzw[0]);
                        item(it + 1, s, n1, n0, d, z1, rxy[W - 1], rzw[W - 1], dxy[W - 1], dzw[W - 1]);
                    } else {
                        item(it, s, cur[it][s], at(bk, o_u[it]), at(bk, o_d[it]), at(bn, o_c[it]), rxy[0], rzw[0],
                             dxy[0], dzw[0]);
                    }
                }
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    if (valid[it + w]) rsum.add(rxy[w], rzw[w]);
                    off[it + w] += DOWN ? 0u - plane : plane;   // modulo 2^32
                }
            }
            // per-thread sums over at most 32 planes, then FP64
            if (!PERIODIC && !EXACT) { lsum0 += lat[0]; lsum1 += lat[1]; }
            if constexpr (EXACT) {   // this plane's densities are in prev now
                if (electrode)
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        CompSum e;
#pragma unroll
                        for (int it = 0; it < IPT; ++it)
                            if (valid[it]) add4(e, prev[it][s]);
                        if (k == 0) flush(1 + s, e.value());
                        if (k == nz - 1) flush(3 + s, e.value());
                    }
            } else {
                if (k == 0) { flush(1, an[0]); flush(2, an[1]); }
                if (k == nz - 1) { flush(3, an[0]); flush(4, an[1]); }
            }
            if (++nacc == 32) {
                flush_sums();
                nacc = 0;
            }
            release(pc);
            pc = pos;
            pos.advance(S);
        }
        flush_sums();
        release(pc);   // the plane zb above the segment
        if (failed) break;
    }
    if (failed && lane == 0) atomicExch(err, 1);
    __syncthreads();
    if (!PROD && tid == 0) {
        // no load may be in flight when the CTA exits: wait (bounded) for the
        // last load issued into each slot (already complete unless a wait
        // was lost)
        for (int j = 0; j < S; ++j)
            if (fills[j] > 0) (void)mbar_wait_bounded(&full[j], (fills[j] - 1u) & 1u);
    }
    if (tid == 0 && !abort_flag) {
        double acc[NQ];
        for (int q = 0; q < NQ; ++q) {
            double t = 0.0;
            for (int w = 0; w < NW; ++w) t += wacc[w * WQ + q];
            acc[q] = t;
        }
        double *sl = slots + (size_t)blockIdx.x * NT;
        sl[0] += acc[0] * cf.rec_f;
        sl[1] += acc[1] * cf.anode_f[0];
        sl[2] += acc[2] * cf.anode_f[1];
        sl[3] += acc[3] * cf.cathode_f[0];
        sl[4] += acc[4] * cf.cathode_f[1];
        // lateral faces: x and y weights are equal for dx = dy (latx_f == laty_f)
        sl[5] += acc[5] * cf.latx_f[0];
        sl[6] += acc[6] * cf.latx_f[1];
        if (SC) {
            sl[7] += acc[NQ - 2] * cf.sc_f[0];
            sl[8] += acc[NQ - 1] * cf.sc_f[1];
        }
    }
}

// The dynamic shared-memory limit is a property of the kernel function,
// shared by every context: raise it to the device's opt-in maximum (never
// lower it to one context's need), so launches of other contexts with
// larger tiles stay valid.
template <bool P, int I, int W, bool S, bool R, bool D, bool E>
static cudaError_t zm_set_attr(size_t smem, int *occ) {
    auto *k = step_zmarch_kernel<P, I, W, S, R, D, E>;
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, k);
    if (e != cudaSuccess) return e;
    const int max_dyn = optin - (int)fa.sharedSizeBytes;   // static shared memory counts against the limit
    if ((int)smem > max_dyn) return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn);
    int n = 0;
    if (e == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, W * 32 + (zm_prod(P, I, S, R) ? 32 : 0), smem) != cudaSuccess)
        n = 0;
    *occ = std::min(*occ, n);
    return e;
}

// both directions of the march (only the upward one with more than two float4
// per thread: the rare shapes whose instances spill)
template <bool P, int I, int W, bool S, bool R, bool E>
static cudaError_t zm_prepare(size_t smem, int *occ) {
    cudaError_t e = zm_set_attr<P, I, W, S, R, false, E>(smem, occ);
    if (I <= 2 && e == cudaSuccess) e = zm_set_attr<P, I, W, S, R, I <= 2, E>(smem, occ);
    return e;
}

// The instance of a launch shape: its shared-memory limit and occupancy, and
// its launch.  The two kinds are instantiated in translation units of their
// own, which compile side by side.
#define ZM_SHAPES(X, S)                                                              \
    X(true, 1, 16, S) X(true, 2, 16, S) X(true, 3, 16, S) X(true, 4, 16, S)          \
    X(false, 1, 16, S) X(false, 2, 16, S) X(false, 3, 16, S) X(false, 4, 16, S)      \
    X(true, 1, 8, S) X(true, 2, 8, S) X(true, 3, 8, S) X(true, 4, 8, S)              \
    X(false, 1, 8, S) X(false, 2, 8, S) X(false, 3, 8, S) X(false, 4, 8, S)

template <bool E>
cudaError_t zm_prepare_shape(bool per, int ipt, int nw, bool sc, bool pair, size_t smem, int *occ) {
    cudaError_t e = cudaSuccess;
#define ZM_CASE(P, I, W, S)                                                                        \
    if (per == P && ipt == I && nw == W && sc == S)                                                \
        e = pair ? zm_prepare<P, I, W, S, I % 2 == 0, E>(smem, occ) : zm_prepare<P, I, W, S, false, E>(smem, occ);
    ZM_SHAPES(ZM_CASE, false)
    ZM_SHAPES(ZM_CASE, true)
#undef ZM_CASE
    return e;
}

template <bool E>
void zm_launch_shape(bool per, int ipt, int nw, bool sc, bool down, int grid, const ZmMaps &maps, const float *ip, const float *im,
                     float *op, float *om,
                     int nx, int ny, int nz, const ZmConf &z, const Coef<float> &cf, double *slots, int *err,
                     cudaStream_t s) {
#define ZM_LAUNCH(P, I, W, S)                                                                              \
    if (per == P && ipt == I && nw == W && sc == S) {                                                      \
        constexpr bool R = I % 2 == 0, D = I <= 2;                                                         \
        auto *k = z.pair ? (down ? step_zmarch_kernel<P, I, W, S, R, D, E>                                 \
                                 : step_zmarch_kernel<P, I, W, S, R, false, E>)                            \
                         : (down ? step_zmarch_kernel<P, I, W, S, false, D, E>                             \
                                 : step_zmarch_kernel<P, I, W, S, false, false, E>);                       \
        k<<<grid, W * 32 + (zm_prod(P, I, S, z.pair) ? 32 : 0), z.smem, s>>>(maps, ip, im, op, om, nx, ny, nz, z,\
                                                                             cf, slots, err);              \
    }
    ZM_SHAPES(ZM_LAUNCH, false)
    ZM_SHAPES(ZM_LAUNCH, true)
#undef ZM_LAUNCH
}

extern template cudaError_t zm_prepare_shape<false>(bool, int, int, bool, bool, size_t, int *);
extern template cudaError_t zm_prepare_shape<true>(bool, int, int, bool, bool, size_t, int *);
extern template void zm_launch_shape<false>(bool, int, int, bool, bool, int, const ZmMaps &, const float *, const float *,
                                            float *, float *, int, int,
                                            int, const ZmConf &, const Coef<float> &, double *, int *, cudaStream_t);
extern template void zm_launch_shape<true>(bool, int, int, bool, bool, int, const ZmMaps &, const float *, const float *,
                                            float *, float *, int, int,
                                           int, const ZmConf &, const Coef<float> &, double *, int *, cudaStream_t);

}  // namespace itk
