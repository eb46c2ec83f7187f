// it_batch.cu -- many independent simulations advanced by one launch per step.
//
// Each simulation is the same method as a single context (Eq. theEquation
// discretised as in the Appendix, deposition of Eqs. linear_density /
// Gaussian / created, electrode tallies and f of Eq. collection_efficiency)
// on its own grid, dx, voltage and time step.  All simulations live in four
// shared FP32 arrays (two ping-pong sets of n+ and n-), each simulation
// aligned to 256 bytes.  Work tables list (simulation, tile or columns, planes)
// entries; one step's launches advance every active simulation by one of its
// own steps, and segments of launches are replayed from a CUDA graph.
// At segment ends the per-entry tally slots are folded into per-simulation
// FP64 accumulators in a fixed order, in-domain charge is measured, and
// finished simulations leave the table.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <string>
#include <vector>

#include "it_device.cuh"
#include "it_internal.cuh"
#include "it_march.cuh"
#include "it_tma.cuh"

namespace itk {

struct BatchSim {
    int nx, ny, nz, pad;
    long long off;          // element offset of this simulation in each state array
    Coef<float> cf;
};

struct BatchEntry {
    int sim, pad;
    long long begin, end;   // row range inside the simulation (row = k * ny + j)
};

// Entry of the marches without a ring: 128 columns (x-segments of four cells,
// or cells) from q0 of one simulation's flattened x-y plane, planes [k0, k1).
struct MarchEntry {
    int sim;
    unsigned q0;
    int k0, k1;
};

// the update weights of a simulation, in registers for the march
struct RegCoef {
    float wx[2], wzm[2], wzp[2], adt, sc[2];
    __device__ __forceinline__ explicit RegCoef(const Coef<float> &c)
        : wx{c.wx[0], c.wx[1]}, wzm{c.wzm[0], c.wzm[1]}, wzp{c.wzp[0], c.wzp[1]}, adt(c.adt), sc{c.sc[0], c.sc[1]} {}
};

// One step of an entry straight from L1/L2 (direct_march with V = 4: the
// simulation's nx % 4 == 0; simple_march with V = 1: any nx): the same
// marches as the single-grid kernels', one unit per block.  Against the
// TMA-staged kernel it has no ring to fill and no tile that is mostly empty:
// per step of surrogate simulations (48 x 48 cells) 256 of them take 136, 64
// 40, 16 12.1 and four 6.3 us, against 166, 60, 20.7 and 16.5 with the ring
// (85, 21, 5.6 and 1.1 at the copy rate); the 256 larger ones of the batched
// workload, which stream from HBM, take 634 against 503.  rev: the entries in
// reverse order (a step of 256 surrogate simulations and their remainders on
// average 62.6 to 59.5 us).
template <bool PERIODIC, bool SC, int V>
__global__ void __launch_bounds__(SK_THREADS, (V == 4 ? DK_BLOCKS : SK_BLOCKS_F32))
step_batched_march_kernel(const BatchSim *__restrict__ sims, const MarchEntry *__restrict__ tab,
                          const float *__restrict__ ip_all, const float *__restrict__ im_all,
                          float *__restrict__ op_all, float *__restrict__ om_all, int rev,
                          double *__restrict__ slots) {
    constexpr int NV = MarchValues<PERIODIC, SC>::N;
    __shared__ double raw[5 * SK_THREADS];
    CompSum(*buf)[SK_THREADS] = reinterpret_cast<CompSum(*)[SK_THREADS]>(raw);
    __shared__ double tot[9];
    const unsigned ent = rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const MarchEntry E = tab[ent];
    const BatchSim &S = sims[E.sim];
    const RegCoef c(S.cf);
    const long long off = S.off;
    if (threadIdx.x < 9) tot[threadIdx.x] = 0.0;
    if constexpr (V == 4)
        direct_march<uint32_t, PERIODIC, SC, false>(ip_all + off, im_all + off, op_all + off, om_all + off, S.nx, S.ny, S.nz,
                                             E.q0, E.k0, E.k1, c, buf, tot);
    else
        simple_march<float, uint32_t, PERIODIC, SC>(ip_all + off, im_all + off, op_all + off, om_all + off, S.nx, S.ny,
                                                    S.nz, E.q0, E.k0, E.k1, c, buf, tot);
    __syncthreads();
    if (threadIdx.x < 9) sk_slot<PERIODIC, SC, NV>(tot, S.cf, slots + (size_t)ent * NT, threadIdx.x, 1);
}

// Entry of the TMA-staged kernel: rows [y0, y0 + rows) of one simulation,
// planes [z0, z1).
struct VecEntry {
    int sim, y0, rows, z0, z1, pad;
};

// TMA-staged float4 z-march over the entries of simulations with nx % 4 == 0
// and nx <= 256: the batched counterpart of the single-context step kernel.
// A CTA owns rows [y0, y0 + rows) of one simulation (full width) and planes
// [z0, z1).  Every plane it needs (z0 - 1 .. z1) arrives by TMA in a ring of
// shared-memory slots: a box of bt = min(IPT floor(256 / (nx/4)), 256, ny)
// rows per species plus one halo row above and below, wrapped when the faces are
// periodic; rows and planes outside the simulation's tensor arrive as zeros
// (the absorbing faces and the electrode ghost planes).  Each simulation's
// tensor maps (two sets x two species x {main box for IPT = 1, main box for
// IPT = 2, halo row}) sit in global memory.  A thread owns IPT float4
// x-segments, two of them one above the other (each is the other's y
// neighbour), keeps planes k-1 and k of them in registers and reads x/y
// neighbours and plane k+1 from shared memory: the same per-cell operation
// sequence as every other kernel.  IPT = 1 runs three CTAs per SM, IPT = 2 two
// with larger rings; a plane's round through the CTA sets the time, and two
// float4 per thread halve the rounds per cell.  With IPT = 2 and no space
// charge a ninth warp refills a slot as soon as its readers have left it;
// otherwise the last warp to release a slot does (the ninth warp leaves 96
// registers per thread).  Steps alternate between the entries' order and its
// reverse.  256 uneven simulations of the batched workload (3.1 GB per step):
// 577 us per step before the pairs and the producer, 503 with them (6.1 TB/s);
// 64 of them: 183 and 158.  Every ring wait is bounded (2^32 SM cycles); a
// wait that runs out raises the error flag, and the CTA drains the copies it
// issued and returns.
constexpr int BT_MAX_S = 8;
constexpr int BT_WARPS = 8;
// dynamic shared memory of the TMA batched kernel with one float4 per thread:
// three CTAs per SM; the ring gets whatever slots fit (3..8; a slot is at
// most 12 KiB at nx = 256)
constexpr int kBtSmem = 70 * 1024;
constexpr int kBtSmemFloats = (kBtSmem - 128) / 4;
// with two float4 per thread: two CTAs per SM, twice the rows per box
constexpr int kBtSmem2 = 105 * 1024;
constexpr int kBtSmemFloats2 = (kBtSmem2 - 128) / 4;
// tensor maps per simulation: [set][species][main box of one float4 per
// thread, main box of two, halo row]
constexpr int BT_MAPS = 12;

__device__ __forceinline__ int bt_align32(int f) { return (f + 31) & ~31; }

__host__ __device__ constexpr bool bt_prod(bool sc, int ipt) { return !sc && ipt == 2; }
__host__ __device__ constexpr int bt_threads(bool sc, int ipt) { return BT_WARPS * 32 + (bt_prod(sc, ipt) ? 32 : 0); }

template <bool PERIODIC, bool SC, int IPT>
__global__ void __launch_bounds__(bt_threads(SC, IPT), (IPT == 1 ? 3 : 2))
step_batched_tma_kernel(const BatchSim *__restrict__ sims, const VecEntry *__restrict__ tab,
                        const CUtensorMap *__restrict__ maps, int parity, float *__restrict__ op_all,
                        float *__restrict__ om_all, double *__restrict__ slots, int smem_floats,
                        int *__restrict__ err) {
    constexpr bool PROD = bt_prod(SC, IPT);
    constexpr int NW = BT_WARPS, WQ = SC ? 16 : 8, NQ = SC ? 9 : 7;
    extern __shared__ __align__(128) unsigned char bt_smem_raw[];
    unsigned char *smem_base = bt_smem_raw + ((128u - (smem_u32(bt_smem_raw) & 127u)) & 127u);
    float *ring = reinterpret_cast<float *>(smem_base);
    __shared__ double wacc[NW * WQ];
    __shared__ __align__(8) uint64_t full[BT_MAX_S];
    __shared__ __align__(8) uint64_t empty[BT_MAX_S];   // PROD: the slot's readers are done with it
    __shared__ uint32_t rel[BT_MAX_S], fills[BT_MAX_S];
    __shared__ volatile int abort_flag;
    __shared__ BatchSim Sm;
    __shared__ VecEntry E;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // steps alternate between the entries' order and its reverse, so that a
    // step first reads what the step before it wrote last (still in L2)
    const unsigned ent = parity ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    if (tid == 0) {
        E = tab[ent];
        Sm = sims[E.sim];
    }
    __syncthreads();
    const int nx = Sm.nx, ny = Sm.ny, nz = Sm.nz;
    const Coef<float> &c = Sm.cf;
    // the weights in registers for the march (read from shared memory at
    // every plane otherwise)
    const float rwx[2] = {c.wx[0], c.wx[1]}, rwzm[2] = {c.wzm[0], c.wzm[1]}, rwzp[2] = {c.wzp[0], c.wzp[1]};
    const float radt = c.adt;
    const int ncol4 = nx >> 2;
    const int bt = min(min(IPT * (256 / ncol4), 256), ny);   // rows of the main box (a box dimension is <= 256)
    const int rows = E.rows;                        // rows computed (<= bt)
    const int reg_main = bt_align32(nx), reg_bot = reg_main + bt_align32(bt * nx), blk = reg_bot + bt_align32(nx);
    const int slotf = 2 * blk;
    const int S = min(smem_floats / slotf, BT_MAX_S);   // the host keeps this >= 3
    const CUtensorMap *mp = maps + (size_t)E.sim * BT_MAPS + parity * 6;   // [species][main1, main2, halo]
    const int z0 = E.z0, z1 = E.z1, y0 = E.y0;
    const int nload = z1 - z0 + 2;                  // planes z0 - 1 .. z1
    const int ytop = PERIODIC ? (y0 > 0 ? y0 - 1 : ny - 1) : y0 - 1;
    const int ybot = PERIODIC ? (y0 + rows < ny ? y0 + rows : 0) : y0 + rows;
    const uint32_t tx = 2u * (uint32_t)(bt + 2) * (uint32_t)nx * 4u;

    // load plane z0 - 1 + n into its slot (one thread)
    auto issue = [&](int n) {
        const int p = z0 - 1 + n;
        const int slot = n % S;
        float *base = ring + (size_t)slot * slotf;
        uint64_t *bar = &full[slot];
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, tx);
        for (int s = 0; s < 2; ++s) {
            float *b = base + s * blk;
            tma_load3(b + reg_main, &mp[3 * s + IPT - 1], bar, 0, y0, p);
            tma_load3(b, &mp[3 * s + 2], bar, 0, ytop, p);
            tma_load3(b + reg_bot, &mp[3 * s + 2], bar, 0, ybot, p);
        }
        fills[slot] += 1;
    };

    if (tid == 0) {
        for (int q = 0; q < 6; ++q) fence_tensormap_acquire(&mp[q]);
        for (int q = 0; q < S; ++q) {
            mbar_init(&full[q], 1);
            if (PROD) mbar_init(&empty[q], NW);
            rel[q] = 0;
            fills[q] = 0;
        }
        for (int q = 0; q < NW * WQ; ++q) wacc[q] = 0.0;
        abort_flag = 0;
        fence_mbar_init();
        for (int n = 0; n < S && n < nload; ++n) issue(n);
    }
    __syncthreads();

    if constexpr (PROD)
        if (warp == NW) {
            // the producer: refills a slot when its readers have left it
            // (bounded wait); no load may be in flight when the CTA exits
            if (lane == 0) {
                RingPos pos{0, 0u};
                for (int n = S; n < nload; ++n) {
                    bool lost = false;
                    if (!mbar_try_wait(&empty[pos.slot], pos.phase)) {
                        const long long t0 = clock64();
                        while (!mbar_try_wait(&empty[pos.slot], pos.phase))
                            if (abort_flag || clock64() - t0 > (1LL << 32)) {
                                lost = true;
                                break;
                            }
                    }
                    if (lost || abort_flag) {
                        abort_flag = 1;
                        atomicExch(err, 1);
                        break;
                    }
                    issue(n);
                    pos.advance(S);
                }
                for (int j = 0; j < S; ++j)
                    if (fills[j] > 0) (void)mbar_wait_bounded(&full[j], (fills[j] - 1u) & 1u);
            }
            __syncwarp();
            __syncthreads();   // the computing warps' last barrier
            return;
        }

    auto flush = [&](int q, float part) {
        double v = (double)part;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) wacc[warp * WQ + q] += v;
    };

    // this thread's float4 segments q = tid + 256 it; threads past the tile
    // repeat its last segment and store nothing
    bool valid[IPT], edge_u[IPT], edge_d[IPT];
    int c4_[IPT], o_c[IPT], o_u[IPT], o_d[IPT], o_l[IPT], o_r[IPT];
    uint32_t off[IPT];
    const uint32_t plane = (uint32_t)nx * (uint32_t)ny;
#pragma unroll
    for (int it = 0; it < IPT; ++it) {
        // two segments: one above the other, so that each is the other's y
        // neighbour (below an odd last row: the halo row, not stored)
        const int q = IPT == 2 ? tid : tid + it * BT_WARPS * 32;
        const int nq = IPT == 2 ? (rows + 1) / 2 * ncol4 : rows * ncol4;
        const int te = q < nq ? q : nq - 1;
        const int tr = te / ncol4, c4 = te - tr * ncol4;
        const int ty = IPT == 2 ? 2 * tr + it : tr;
        valid[it] = q < nq && ty < rows;
        const int x0 = 4 * c4;
        c4_[it] = c4;
        o_c[it] = ty < rows ? reg_main + ty * nx + x0 : reg_bot + x0;
        o_u[it] = ty == 0 ? x0 : reg_main + (ty - 1) * nx + x0;
        o_d[it] = ty >= rows - 1 ? reg_bot + x0 : reg_main + (ty + 1) * nx + x0;
        o_l[it] = reg_main + ty * nx + (c4 == 0 ? nx - 1 : x0 - 1);
        o_r[it] = reg_main + ty * nx + (c4 == ncol4 - 1 ? 0 : x0 + 4);
        const int yg = y0 + ty;
        edge_u[it] = !PERIODIC && yg == 0;
        edge_d[it] = !PERIODIC && yg == ny - 1;
        off[it] = ((uint32_t)z0 * (uint32_t)ny + (uint32_t)yg) * (uint32_t)nx + (uint32_t)x0;
    }
    float *out_[2] = {op_all + Sm.off, om_all + Sm.off};

    RingPos pos{0, 0u};
    int nrel = 0;
    bool failed = false;
    auto wait_full = [&](const RingPos &u) {
        if (failed) return;
        bool ok = mbar_try_wait(&full[u.slot], u.phase);
        if (__all_sync(0xffffffffu, ok)) return;
        const long long t0 = clock64();
        for (;;) {
            ok = ok || mbar_try_wait(&full[u.slot], u.phase);
            if (__all_sync(0xffffffffu, ok)) return;
            if (__any_sync(0xffffffffu, abort_flag || clock64() - t0 > (1LL << 32))) break;
        }
        failed = true;
        if (lane == 0) abort_flag = 1;
    };
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

    float4 prev[IPT][2], cur[IPT][2];
    wait_full(pos);
    {
        const float *sl = ring + (size_t)pos.slot * slotf;
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            prev[it][0] = *reinterpret_cast<const float4 *>(sl + o_c[it]);
            prev[it][1] = *reinterpret_cast<const float4 *>(sl + blk + o_c[it]);
        }
    }
    release(pos);
    pos.advance(S);
    wait_full(pos);
    RingPos pc = pos;
    pos.advance(S);
    {
        const float *sl = ring + (size_t)pc.slot * slotf;
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            cur[it][0] = *reinterpret_cast<const float4 *>(sl + o_c[it]);
            cur[it][1] = *reinterpret_cast<const float4 *>(sl + blk + o_c[it]);
        }
    }
    float rsum = 0.f, lsum0 = 0.f, lsum1 = 0.f, ssum0 = 0.f, ssum1 = 0.f;
    int nacc = 0;
    for (int k = z0; k < z1; ++k) {
        wait_full(pos);
        const float *sk = ring + (size_t)pc.slot * slotf;
        const float *sn = ring + (size_t)pos.slot * slotf;
        float an[2] = {0.f, 0.f}, lat[2] = {0.f, 0.f};
        float2 rxy[IPT], rzw[IPT], dxy[IPT], dzw[IPT];
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            const float4 P = cur[it][0], M = cur[it][1];
            rxy[it] = __fmul2_rn(make_float2(P.x, P.y), make_float2(M.x, M.y));
            rzw[it] = __fmul2_rn(make_float2(P.z, P.w), make_float2(M.z, M.w));
            if (SC) sc_diff4(P, M, dxy[it], dzw[it]);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const float *bk = sk + s * blk;
            auto at = [](const float *q, int o) { return *reinterpret_cast<const float4 *>(q + o); };
            const float4 above = at(bk, o_u[0]), below = at(bk, o_d[IPT - 1]);
            float4 nc[IPT];
#pragma unroll
            for (int it = 0; it < IPT; ++it) nc[it] = cur[it][s];
#pragma unroll
            for (int it = 0; it < IPT; ++it) {
                const float4 n = nc[it];
                const float4 u = it == 0 ? above : nc[0], d = it == IPT - 1 ? below : nc[IPT - 1];
                const float4 zp = at(sn + s * blk, o_c[it]);
                float l = bk[o_l[it]];
                float r = bk[o_r[it]];
                if (!PERIODIC) {
                    if (c4_[it] == 0) l = 0.f;
                    if (c4_[it] == ncol4 - 1) r = 0.f;
                }
                float4 v = upd7x4(n, l, r, u, d, prev[it][s], zp, rxy[it], rzw[it], rwx[s], rwzm[s], rwzp[s], radt);
                if (SC) {
                    float2 pxy, pzw;
                    v = add_sc4(v, c.sc[s], n, dxy[it], dzw[it], pxy, pzw);
                    if (valid[it]) (s ? ssum1 : ssum0) += (pxy.x + pxy.y) + (pzw.x + pzw.y);
                }
                if (valid[it]) {
                    *reinterpret_cast<float4 *>(out_[s] + off[it]) = v;
                    if (k == 0 || k == nz - 1) an[s] += (n.x + n.y) + (n.z + n.w);
                    if (!PERIODIC) {
                        if (c4_[it] == 0) lat[s] += n.x;
                        if (c4_[it] == ncol4 - 1) lat[s] += n.w;
                        if (edge_u[it]) lat[s] += (n.x + n.y) + (n.z + n.w);
                        if (edge_d[it]) lat[s] += (n.x + n.y) + (n.z + n.w);
                    }
                }
                prev[it][s] = n;
                cur[it][s] = zp;
            }
        }
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            if (valid[it]) rsum += (rxy[it].x + rxy[it].y) + (rzw[it].x + rzw[it].y);
            off[it] += plane;
        }
        if (!PERIODIC) { lsum0 += lat[0]; lsum1 += lat[1]; }
        if (++nacc == 32) {
            flush(0, rsum);
            rsum = 0.f;
            if (!PERIODIC) { flush(5, lsum0); flush(6, lsum1); lsum0 = lsum1 = 0.f; }
            if (SC) { flush(7, ssum0); flush(8, ssum1); ssum0 = ssum1 = 0.f; }
            nacc = 0;
        }
        if (k == 0) { flush(1, an[0]); flush(2, an[1]); }
        if (k == nz - 1) { flush(3, an[0]); flush(4, an[1]); }
        release(pc);
        pc = pos;
        pos.advance(S);
    }
    flush(0, rsum);
    if (!PERIODIC) { flush(5, lsum0); flush(6, lsum1); }
    if (SC) { flush(7, ssum0); flush(8, ssum1); }
    release(pc);   // plane z1
    if (failed && lane == 0) atomicExch(err, 1);
    __syncthreads();
    if (!PROD && tid == 0) {
        // no copy may be in flight when the CTA exits
        for (int j = 0; j < S; ++j)
            if (fills[j] > 0) (void)mbar_wait_bounded(&full[j], (fills[j] - 1u) & 1u);
    }
    if (tid == 0 && !abort_flag) {
        double acc[NQ];
        for (int q = 0; q < NQ; ++q) {
            double v = 0.0;
            for (int w = 0; w < NW; ++w) v += wacc[w * WQ + q];
            acc[q] = v;
        }
        double *sl = slots + (size_t)ent * NT;
        sl[0] += acc[0] * c.rec_f;
        sl[1] += acc[1] * c.anode_f[0];
        sl[2] += acc[2] * c.anode_f[1];
        sl[3] += acc[3] * c.cathode_f[0];
        sl[4] += acc[4] * c.cathode_f[1];
        sl[5] += acc[5] * c.latx_f[0];
        sl[6] += acc[6] * c.latx_f[1];
        if (SC) {
            sl[7] += acc[NQ - 2] * c.sc_f[0];
            sl[8] += acc[NQ - 1] * c.sc_f[1];
        }
    }
}

// Fold the slots of each active simulation's entries (contiguous in the
// table, in order) into its FP64 accumulators and clear them.  One block per
// active simulation, one warp per tally.
__global__ void __launch_bounds__(NT * 32)
batch_fold_kernel(const int *__restrict__ first, const int *__restrict__ count, const int *__restrict__ sim_of,
                  double *__restrict__ slots, double *__restrict__ acc) {
    const int a = blockIdx.x, lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    double *sl = slots + (size_t)first[a] * NT;
    const int n = count[a];
    const double s = warp_strided_sum(sl, n, q, NT, lane);
    for (int e = lane; e < n; e += 32) sl[(size_t)e * NT + q] = 0.0;
    if (lane == 0) acc[(size_t)sim_of[a] * NT + q] += s;
}

// Per-entry sums of n+ and n- for the in-domain charge, and their largest
// value for the dt ladder: FP32 partials over at most 32 cells per thread,
// then FP64 (once per 32 cells, outside the per-cell loop: FP64 arithmetic is
// slow on this GPU).
__global__ void __launch_bounds__(256)
batch_monitor_kernel(const BatchSim *__restrict__ sims, const BatchEntry *__restrict__ tab,
                     const float *__restrict__ ip_all, const float *__restrict__ im_all, double *__restrict__ mon) {
    __shared__ double red[32 * 2];
    __shared__ float rmax[8];
    const BatchEntry E = tab[blockIdx.x];
    const long long off = sims[E.sim].off;
    const long long nxs = sims[E.sim].nx;
    double v[2] = {0.0, 0.0};
    float mx = -INFINITY;
    const size_t end = (size_t)(E.end * nxs);
    size_t idx = (size_t)(E.begin * nxs) + threadIdx.x;
    while (idx < end) {
        float a = 0.f, b = 0.f;
        for (int j = 0; j < 32 && idx < end; ++j, idx += blockDim.x) {
            const float p = ip_all[off + idx], m = im_all[off + idx];
            a += p;
            b += m;
            mx = fmaxf(mx, fmaxf(p, m));
        }
        v[0] += (double)a;
        v[1] += (double)b;
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) rmax[threadIdx.x >> 5] = mx;
    block_sum<2>(v, red);   // contains the __syncthreads for rmax too
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) mx = fmaxf(mx, rmax[w]);
        mon[3 * blockIdx.x] = v[0];
        mon[3 * blockIdx.x + 1] = v[1];
        mon[3 * blockIdx.x + 2] = (double)mx;
    }
}

// One simulation's results in one place: out[0 .. NT) tallies, two released
// charges, two in-domain sums, two smallest and two largest densities.  One
// warp per value.
constexpr int TAL_BLOCKS = 64, TAL_OUT = NT + 8;
__global__ void __launch_bounds__(TAL_OUT * 32)
batch_tally_kernel(const double *__restrict__ acc, const double *__restrict__ rel, const double *__restrict__ mon,
                   double *__restrict__ out) {
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    double v = 0.0;
    if (q < NT) {
        v = acc[q];
    } else if (q < NT + 2) {
        v = rel[q - NT];
    } else if (q < NT + 4) {
        v = warp_strided_sum(mon, TAL_BLOCKS, q - NT - 2, NM, lane);
    } else {
        const int e = q - NT - 2;   // 2, 3 smallest, 4, 5 largest
        v = e < 4 ? INFINITY : -INFINITY;
        for (int m = lane; m < TAL_BLOCKS; m += 32) {
            const double x = mon[(size_t)m * NM + e];
            v = e < 4 ? fmin(v, x) : fmax(v, x);
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double x = __shfl_down_sync(0xffffffffu, v, o);
            v = e < 4 ? fmin(v, x) : fmax(v, x);
        }
    }
    if (lane == 0) out[q] = v;
}

// Per-entry maximum of n+ and n-.
__global__ void __launch_bounds__(256)
batch_max_kernel(const BatchSim *__restrict__ sims, const BatchEntry *__restrict__ tab,
                 const float *__restrict__ ip_all, const float *__restrict__ im_all, float *__restrict__ mx) {
    __shared__ float red[32];
    const BatchEntry E = tab[blockIdx.x];
    const long long off = sims[E.sim].off;
    const long long nxs = sims[E.sim].nx;
    float v = -INFINITY;
    for (size_t idx = (size_t)(E.begin * nxs) + threadIdx.x; idx < (size_t)(E.end * nxs); idx += blockDim.x)
        v = fmaxf(v, fmaxf(ip_all[off + idx], im_all[off + idx]));
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = fmaxf(v, red[w]);
        mx[blockIdx.x] = v;
    }
}

// Launch shape of a step for the simulations with nx % 4 == 0.
struct BatchShape {
    int tma;   // 2 / 1: TMA-staged kernel with two / one float4 per thread; 0: direct march
    int cps;   // TMA: CTAs per SM its z splits aim for; direct: divisor of the fitted chunk length
};

}  // namespace itk

using namespace itk;

struct it_batch {
    int nsim;
    it_params p;
    std::vector<it_sim_desc> desc;
    std::vector<BatchSim> hs;         // host copy of the descriptors
    std::vector<double> dx;
    std::vector<double> dt;
    size_t total;                     // elements per state array
    float *state[2][2];               // [set][species]
    void *state_base;
    BatchSim *d_sims;
    double *d_acc;                    // [nsim][NT] folded tallies
    double *d_rel;                    // [nsim][8] released (DevAcc layout)
    // work tables of the current segment
    std::vector<BatchEntry> tab;      // row ranges of every active simulation (monitors)
    std::vector<int> mfirst, mcount;  // per active simulation, into tab
    std::vector<int> morder;          // the active simulation of each mfirst/mcount entry
    std::vector<VecEntry> vtab;       // step entries of the TMA-staged kernel
    std::vector<MarchEntry> dtab;     // of the direct march (float4 segments)
    std::vector<MarchEntry> stab;     // of the march over single cells (nx % 4 != 0)
    std::vector<int> first, count, sim_of;   // per active simulation, into the step slots
    BatchEntry *d_tab;
    VecEntry *d_vtab;
    MarchEntry *d_dtab, *d_stab;
    int *d_first, *d_count, *d_simof;
    double *d_slots, *d_mon;
    std::vector<double> nmax;         // per simulation: largest density at the last check
    size_t tab_cap, stab_cap, dtab_cap, vtab_cap, slot_cap, act_cap;
    long long chunk;                  // cells per entry (monitors, single-cell march)
    BatchShape shape;                 // launch shape of the current table
    bool tuned;                       // the autotuner's choice, for the simulations it was made for
    BatchShape tuned_shape;
    int tuned_active;
    bool forced;                      // test hook: forced_shape whatever is active
    BatchShape forced_shape;
    double cal[3];                    // measured over fitted time of the direct march and the TMA kernels
    double *d_tal;                    // one simulation's monitor blocks, then its gathered tallies
    // per simulation
    std::vector<int64_t> steps;
    std::vector<double> t_s;          // simulated time: the sum of every step's dt
    std::vector<char> active;
    int64_t bstep;                    // steps taken by every active simulation
    cudaStream_t stream;
    cudaGraphExec_t graph;
    int graph_len, graph_parity;
    bool tab_dirty;
    double active_bytes;   // both sets of the simulations in the tables
    // pulse trains: each simulation's deposited tracks are re-deposited every
    // period_steps steps until count pulses have been released
    std::vector<std::vector<double>> pulse_tracks;   // packed [n][4]
    std::vector<int32_t> pulse_count, pulse_done;
    std::vector<int64_t> pulse_period;
    // deposition scratch (sized for the largest simulation)
    double *d_plane, *d_tracks, *d_wx, *d_wy;
    int64_t track_cap;
    int max_nx, max_ny;
    // TMA-staged float4 kernel: per simulation [set][species][main, halo]
    // tensor maps (zero for simulations it does not take) and the device error
    // flag of its bounded waits
    CUtensorMap *d_maps;
    std::vector<char> tma_ok;
    int *d_err;
};

namespace {

int bfail(int code, const std::string &m) {
    set_error(m);
    return code;
}

int sm_count() {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

int tma_rows(const BatchSim &h, int ipt) { return std::max(1, std::min(ipt * (256 / (h.nx / 4)), 256)); }
long long march_blocks(const BatchSim &h, int v) {
    return ((long long)(h.nx / v) * h.ny + SK_THREADS - 1) / SK_THREADS;
}

// z splits of the TMA entries: about cps CTAs per SM, at least eight planes each
int tma_split(const it_batch *b, const BatchShape &sh, int sms) {
    long long tiles = 0;
    for (int s = 0; s < b->nsim; ++s)
        if (b->active[s] && b->tma_ok[s]) {
            const int rows = tma_rows(b->hs[s], sh.tma);
            tiles += (b->hs[s].ny + rows - 1) / rows;
        }
    return tiles > 0 ? (int)std::max(1LL, ((long long)sh.cps * sms + tiles - 1) / tiles) : 1;
}

// Planes per entry of the direct march and its fitted time in us: the blocks
// resident at a time walk their planes in 650 cycles plus 190 per block they
// share the SM with (the single-grid march's figures), an entry starting with
// two planes of loads; a state beyond L2 moves 1.42 times slower than a copy.
int direct_chunk(const it_batch *b, int sms, double *us) {
    const double resident = (double)sms * DK_BLOCKS;
    int best = 1;
    double best_cost = 1e300, bytes = 0.0;
    for (int kc : {1, 2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32, 48, 64, 96, 128, 256, 512}) {
        double entries = 0.0, work = 0.0;
        int longest = 0;
        bytes = 0.0;
        for (int s = 0; s < b->nsim; ++s) {
            const BatchSim &h = b->hs[s];
            if (!b->active[s] || h.nx % 4 != 0) continue;
            const int c = (h.nz + kc - 1) / kc;
            const double nb = (double)march_blocks(h, 4);
            entries += nb * c;
            work += nb * (h.nz + 2.0 * c);
            longest = std::max(longest, (h.nz + c - 1) / c);
            bytes += 16.0 * h.nx * h.ny * h.nz;
        }
        const double full = DK_LAT + DK_THR * DK_BLOCKS;
        const double cost = entries <= resident
                                ? (longest + 2.0) * (DK_LAT + DK_THR * std::ceil(entries / sms))
                                : work / resident * full + 0.5 * (longest + 2.0) * full;
        if (cost < best_cost) {
            best_cost = cost;
            best = kc;
        }
    }
    *us = std::max(best_cost / 1900.0 + 1.5, bytes > 100e6 ? 1.42 * bytes / 6.8e6 : 0.0);
    return best;
}

// Fitted time of a step of the active simulations in us, TMA-staged: a plane's
// round takes 1.3 us with two float4 per thread and two CTAs per SM (1.5 with
// space charge, which has no producer warp), 1.32 with one and three, the last
// entries leave the chip a fifth of the longest one idle, and starting takes
// about 6 us (256 uneven simulations of the batched workload at one, two,
// three and six z splits: 552, 510, 503 and 531 us, fitted 537, 519, 519 and
// 534; 64 of them at three, five and ten: 163, 158 and 170, fitted 159, 156
// and 160).
double tma_us(const it_batch *b, const BatchShape &sh, int sms) {
    const int split = tma_split(b, sh, sms);
    const double round = sh.tma == 2 ? (b->p.space_charge ? 1.5 : 1.3) : 1.32;
    double rounds = 0.0;
    int longest = 0;
    for (int s = 0; s < b->nsim; ++s) {
        const BatchSim &h = b->hs[s];
        if (!b->active[s] || !b->tma_ok[s]) continue;
        const int rows = tma_rows(h, sh.tma), zc = std::min(split, std::max(1, h.nz / 8));
        rounds += (double)((h.ny + rows - 1) / rows) * (h.nz + 2.0 * zc);
        longest = std::max(longest, (h.nz + zc - 1) / zc);
    }
    return rounds * round / ((sh.tma == 2 ? 2.0 : 3.0) * sms) + 0.2 * (longest + 2) * round + 6.0;
}

double shape_us(const it_batch *b, const BatchShape &sh, int sms) {
    double us = 0.0;
    if (sh.tma == 0) (void)direct_chunk(b, sms, &us);
    else us = tma_us(b, sh, sms);
    return us;
}

// The launch shape for the simulations now active: the autotuner's while they
// are the ones it timed, else the least fitted time, scaled by what the
// autotuner measured against the fit (batches shrink as simulations finish,
// and small ones are faster without the ring).
BatchShape choose_shape(const it_batch *b, int sms) {
    int active = 0;
    bool any_tma = false;
    for (int s = 0; s < b->nsim; ++s)
        if (b->active[s]) {
            ++active;
            any_tma = any_tma || b->tma_ok[s];
        }
    if (b->forced) return b->forced_shape;
    if (b->tuned && active == b->tuned_active) return b->tuned_shape;
    BatchShape best{0, 1};
    double best_us = shape_us(b, best, sms) * b->cal[0];
    if (any_tma)
        for (int tma : {2, 1})
            for (int cps : {1, 2, 4, 8, 16, 32}) {
                const BatchShape sh{tma, cps};
                const double us = tma_us(b, sh, sms) * b->cal[tma];
                if (us < best_us) {
                    best_us = us;
                    best = sh;
                }
            }
    return best;
}

// Rebuild the work tables for the active simulations in launch shape b->shape.
// All step entries of one simulation are contiguous, so the fold is in order.
int build_table(it_batch *b) {
    b->tab.clear(); b->mfirst.clear(); b->mcount.clear(); b->morder.clear();
    b->vtab.clear(); b->dtab.clear(); b->stab.clear();
    b->first.clear(); b->count.clear(); b->sim_of.clear();
    long long active_cells = 0;
    for (int s = 0; s < b->nsim; ++s)
        if (b->active[s]) active_cells += (long long)b->hs[s].nx * b->hs[s].ny * b->hs[s].nz;
    b->active_bytes = 16.0 * (double)active_cells;
    const int sms = sm_count();
    const long long chunk = std::max(1024LL, std::min(b->chunk, active_cells / (4LL * sms)));
    const BatchShape sh = b->shape;
    const int split = sh.tma ? tma_split(b, sh, sms) : 1;
    double us = 0.0;
    const int kc4 = std::max(1, direct_chunk(b, sms, &us) / (sh.tma ? 1 : sh.cps));
    const int kc1 = (int)std::max(1LL, chunk / SK_THREADS);
    std::vector<int> part[3], pfirst[3], pcount[3];   // simulations on the TMA, direct and single-cell kernels
    auto march = [&](std::vector<MarchEntry> &tab, int s, int v, int kc) {
        const BatchSim &h = b->hs[s];
        const int c = (h.nz + kc - 1) / kc;
        const long long nb = march_blocks(h, v);
        for (int q = 0; q < c; ++q)
            for (long long p = 0; p < nb; ++p)
                tab.push_back(MarchEntry{s, (unsigned)(p * SK_THREADS), (int)((long long)h.nz * q / c),
                                         (int)((long long)h.nz * (q + 1) / c)});
    };
    for (int s = 0; s < b->nsim; ++s) {
        if (!b->active[s]) continue;
        const BatchSim &h = b->hs[s];
        const long long rows = (long long)h.ny * h.nz;
        const long long rpe = std::max(1LL, chunk / h.nx);
        b->mfirst.push_back((int)b->tab.size());
        int n = 0;
        for (long long r0 = 0; r0 < rows; r0 += rpe, ++n) b->tab.push_back(BatchEntry{s, 0, r0, std::min(rows, r0 + rpe)});
        b->mcount.push_back(n);
        b->morder.push_back(s);
        const int on = h.nx % 4 != 0 ? 2 : sh.tma && b->tma_ok[s] ? 0 : 1;
        const size_t before = on == 0 ? b->vtab.size() : on == 1 ? b->dtab.size() : b->stab.size();
        if (on == 0) {
            // rows per entry: a 256-thread tile of float4 times those per thread
            const int rpt = tma_rows(h, sh.tma);
            const int zc = std::min(split, std::max(1, h.nz / 8));
            for (int y0 = 0; y0 < h.ny; y0 += rpt)
                for (int q = 0; q < zc; ++q)
                    b->vtab.push_back(VecEntry{s, y0, std::min(rpt, h.ny - y0), (int)((long long)h.nz * q / zc),
                                               (int)((long long)h.nz * (q + 1) / zc), 0});
        } else if (on == 1) {
            march(b->dtab, s, 4, kc4);
        } else {
            march(b->stab, s, 1, kc1);
        }
        const size_t after = on == 0 ? b->vtab.size() : on == 1 ? b->dtab.size() : b->stab.size();
        part[on].push_back(s);
        pfirst[on].push_back((int)before);
        pcount[on].push_back((int)(after - before));
    }
    // step slots: [TMA entries][direct entries][single-cell entries]
    const int base[3] = {0, (int)b->vtab.size(), (int)(b->vtab.size() + b->dtab.size())};
    for (int on = 0; on < 3; ++on)
        for (size_t q = 0; q < part[on].size(); ++q) {
            b->sim_of.push_back(part[on][q]);
            b->first.push_back(base[on] + pfirst[on][q]);
            b->count.push_back(pcount[on][q]);
        }
    const size_t ne = b->tab.size(), nvs = b->vtab.size(), nds = b->dtab.size(), nss = b->stab.size(), na = b->sim_of.size();
    const size_t nslot = nvs + nds + nss;
    auto grow = [&](void **p, size_t &cap, size_t need, size_t esz) -> cudaError_t {
        if (need <= cap) return cudaSuccess;
        cudaFree(*p);
        *p = nullptr;
        cap = 0;
        cudaError_t e = cudaMalloc(p, esz * need);
        if (e == cudaSuccess) cap = need;
        return e;
    };
    size_t mon_cap = b->tab_cap;
    IT_CK(grow((void **)&b->d_tab, b->tab_cap, ne, sizeof(BatchEntry)));
    if (b->tab_cap != mon_cap || !b->d_mon) {
        cudaFree(b->d_mon);
        b->d_mon = nullptr;
        IT_CK(cudaMalloc(&b->d_mon, sizeof(double) * 3 * std::max<size_t>(b->tab_cap, 1)));
    }
    IT_CK(grow((void **)&b->d_vtab, b->vtab_cap, nvs, sizeof(VecEntry)));
    IT_CK(grow((void **)&b->d_dtab, b->dtab_cap, nds, sizeof(MarchEntry)));
    IT_CK(grow((void **)&b->d_stab, b->stab_cap, nss, sizeof(MarchEntry)));
    IT_CK(grow((void **)&b->d_slots, b->slot_cap, nslot, sizeof(double) * NT));
    if (na > b->act_cap) {
        cudaFree(b->d_first); cudaFree(b->d_count); cudaFree(b->d_simof);
        IT_CK(cudaMalloc(&b->d_first, sizeof(int) * na));
        IT_CK(cudaMalloc(&b->d_count, sizeof(int) * na));
        IT_CK(cudaMalloc(&b->d_simof, sizeof(int) * na));
        b->act_cap = na;
    }
    if (ne) IT_CK(cudaMemcpyAsync(b->d_tab, b->tab.data(), sizeof(BatchEntry) * ne, cudaMemcpyHostToDevice, b->stream));
    if (nvs) IT_CK(cudaMemcpyAsync(b->d_vtab, b->vtab.data(), sizeof(VecEntry) * nvs, cudaMemcpyHostToDevice, b->stream));
    if (nds) IT_CK(cudaMemcpyAsync(b->d_dtab, b->dtab.data(), sizeof(MarchEntry) * nds, cudaMemcpyHostToDevice, b->stream));
    if (nss) IT_CK(cudaMemcpyAsync(b->d_stab, b->stab.data(), sizeof(MarchEntry) * nss, cudaMemcpyHostToDevice, b->stream));
    if (nslot) IT_CK(cudaMemsetAsync(b->d_slots, 0, sizeof(double) * NT * nslot, b->stream));
    if (na) {
        IT_CK(cudaMemcpyAsync(b->d_first, b->first.data(), sizeof(int) * na, cudaMemcpyHostToDevice, b->stream));
        IT_CK(cudaMemcpyAsync(b->d_count, b->count.data(), sizeof(int) * na, cudaMemcpyHostToDevice, b->stream));
        IT_CK(cudaMemcpyAsync(b->d_simof, b->sim_of.data(), sizeof(int) * na, cudaMemcpyHostToDevice, b->stream));
    }
    IT_CK(cudaStreamSynchronize(b->stream));   // host vectors may change at the next rebuild
    if (b->graph) { cudaGraphExecDestroy(b->graph); b->graph = nullptr; }
    b->tab_dirty = false;
    return IT_OK;
}

// the tables in the launch shape chosen for the active simulations
int rebuild(it_batch *b) {
    b->shape = choose_shape(b, sm_count());
    return build_table(b);
}

int launch_batched_step(it_batch *b, int parity) {
    const int nt = (int)b->vtab.size(), nd = (int)b->dtab.size(), ns = (int)b->stab.size();
    const float *ip = b->state[parity][0], *im = b->state[parity][1];
    float *op = b->state[parity ^ 1][0], *om = b->state[parity ^ 1][1];
    const bool per = b->p.lateral_bc == IT_PERIODIC;
    const bool sc = b->p.space_charge != 0;
    // alternating order of the entries where the state streams from HBM
    const int rev = parity && b->active_bytes > DK_ALTERNATE;
    if (nt) {
        const bool two = b->shape.tma == 2;
        auto *kt = two ? (per ? (sc ? step_batched_tma_kernel<true, true, 2> : step_batched_tma_kernel<true, false, 2>)
                              : (sc ? step_batched_tma_kernel<false, true, 2> : step_batched_tma_kernel<false, false, 2>))
                       : (per ? (sc ? step_batched_tma_kernel<true, true, 1> : step_batched_tma_kernel<true, false, 1>)
                              : (sc ? step_batched_tma_kernel<false, true, 1> : step_batched_tma_kernel<false, false, 1>));
        kt<<<nt, bt_threads(sc, two ? 2 : 1), two ? kBtSmem2 : kBtSmem, b->stream>>>(b->d_sims, b->d_vtab, b->d_maps, parity, op,
                                                                       om, b->d_slots,
                                                                       two ? kBtSmemFloats2 : kBtSmemFloats, b->d_err);
        IT_CK(cudaGetLastError());
    }
    if (nd) {
        auto *kd = per ? (sc ? step_batched_march_kernel<true, true, 4> : step_batched_march_kernel<true, false, 4>)
                       : (sc ? step_batched_march_kernel<false, true, 4> : step_batched_march_kernel<false, false, 4>);
        kd<<<nd, SK_THREADS, 0, b->stream>>>(b->d_sims, b->d_dtab, ip, im, op, om, rev,
                                                b->d_slots + (size_t)NT * nt);
        IT_CK(cudaGetLastError());
    }
    if (ns) {
        auto *ks = per ? (sc ? step_batched_march_kernel<true, true, 1> : step_batched_march_kernel<true, false, 1>)
                       : (sc ? step_batched_march_kernel<false, true, 1> : step_batched_march_kernel<false, false, 1>);
        ks<<<ns, SK_THREADS, 0, b->stream>>>(b->d_sims, b->d_stab, ip, im, op, om, rev,
                                                b->d_slots + (size_t)NT * (nt + nd));
        IT_CK(cudaGetLastError());
    }
    return IT_OK;
}

// K steps of every active simulation (K even: the graph returns to the same set)
int run_segment(it_batch *b, int K) {
    const int parity = (int)(b->bstep & 1);
    if (!b->graph || b->graph_len != K || b->graph_parity != parity) {
        if (b->graph) { cudaGraphExecDestroy(b->graph); b->graph = nullptr; }
        cudaGraph_t g = nullptr;
        IT_CK(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
        int rc = IT_OK;
        for (int q = 0; q < K && rc == IT_OK; ++q) rc = launch_batched_step(b, parity ^ (q & 1));
        cudaError_t e = cudaStreamEndCapture(b->stream, &g);
        if (rc) { if (g) cudaGraphDestroy(g); return rc; }
        if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture(batch)");
        e = cudaGraphInstantiate(&b->graph, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) { b->graph = nullptr; return cuda_fail(e, "cudaGraphInstantiate(batch)"); }
        b->graph_len = K;
        b->graph_parity = parity;
    }
    IT_CK(cudaGraphLaunch(b->graph, b->stream));
    b->bstep += K;
    for (int s = 0; s < b->nsim; ++s)
        if (b->active[s]) {
            b->steps[s] += K;
            b->t_s[s] += b->dt[s] * K;
        }
    return IT_OK;
}

// The doubling ladder of it_run_to_completion, per active simulation with no
// pulse still to come: its dt rises to the largest rung admissible at the
// peak density the check has just measured.  The step graph reads the
// descriptors from device memory, so only they change.
static int ladder_batch(it_batch *b) {
    for (size_t a = 0; a < b->morder.size(); ++a) {
        const int s = b->morder[a];
        const double nmax = b->nmax[s];
        // as in a single context, whose check runs before the deposits of its
        // step: a check at the step of the last pulse still counts that pulse
        // as to come
        const bool last_now = b->pulse_count[s] > 1 && b->pulse_done[s] == b->pulse_count[s] &&
                              b->steps[s] == (int64_t)(b->pulse_count[s] - 1) * b->pulse_period[s];
        const bool pending = (b->pulse_done[s] >= 1 && b->pulse_done[s] < b->pulse_count[s]) || last_now;
        if (pending) continue;
        const it_sim_desc &d = b->desc[s];
        it_params p = b->p;
        p.gap_cm = d.nz * d.dx_cm;
        p.voltage_V = d.voltage_V;
        const double nd = ladder_rung(&p, d.dx_cm, b->dt[s], nmax);
        if (nd > b->dt[s]) {
            b->dt[s] = nd;
            coef_f32(&p, d.dx_cm, nd, &b->hs[s].cf);
            IT_CK(cudaMemcpyAsync(b->d_sims + s, &b->hs[s], sizeof(BatchSim), cudaMemcpyHostToDevice, b->stream));
        }
    }
    IT_CK(cudaStreamSynchronize(b->stream));
    return IT_OK;
}

int fold(it_batch *b) {
    const int na = (int)b->sim_of.size();
    if (!na) return IT_OK;
    batch_fold_kernel<<<na, NT * 32, 0, b->stream>>>(b->d_first, b->d_count, b->d_simof, b->d_slots, b->d_acc);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// in-domain ions of every simulation in the current table, and its largest density
int in_domain(it_batch *b, std::vector<double> &ind2) {
    ind2.assign(2 * (size_t)b->nsim, 0.0);
    const int ne = (int)b->tab.size();
    if (!ne) return IT_OK;
    const int parity = (int)(b->bstep & 1);
    batch_monitor_kernel<<<ne, 256, 0, b->stream>>>(b->d_sims, b->d_tab, b->state[parity][0], b->state[parity][1],
                                                    b->d_mon);
    IT_CK(cudaGetLastError());
    std::vector<double> mon(3 * (size_t)ne);
    int err = 0;
    IT_CK(cudaMemcpyAsync(mon.data(), b->d_mon, sizeof(double) * 3 * ne, cudaMemcpyDeviceToHost, b->stream));
    IT_CK(cudaMemcpyAsync(&err, b->d_err, sizeof(int), cudaMemcpyDeviceToHost, b->stream));
    IT_CK(cudaStreamSynchronize(b->stream));
    if (err) return bfail(IT_ETIMEOUT, "a bounded device wait ran out in the batched step kernel");
    for (size_t a = 0; a < b->morder.size(); ++a) {
        const int s = b->morder[a];
        const double vol = b->dx[s] * b->dx[s] * b->dx[s];
        double p = 0, m = 0, mx = -INFINITY;
        for (int e = b->mfirst[a]; e < b->mfirst[a] + b->mcount[a]; ++e) {
            p += mon[3 * e];
            m += mon[3 * e + 1];
            mx = std::max(mx, mon[3 * e + 2]);
        }
        b->nmax[s] = mx;
        ind2[2 * s] = p * vol;
        ind2[2 * s + 1] = m * vol;
    }
    return IT_OK;
}

void batch_free(it_batch *b) {
    if (!b) return;
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    cudaFree(b->state_base);
    cudaFree(b->d_sims); cudaFree(b->d_acc); cudaFree(b->d_rel);
    cudaFree(b->d_tab); cudaFree(b->d_slots); cudaFree(b->d_mon); cudaFree(b->d_tal);
    cudaFree(b->d_vtab); cudaFree(b->d_dtab); cudaFree(b->d_stab);
    cudaFree(b->d_first); cudaFree(b->d_count); cudaFree(b->d_simof);
    cudaFree(b->d_plane); cudaFree(b->d_tracks); cudaFree(b->d_wx); cudaFree(b->d_wy);
    cudaFree(b->d_maps); cudaFree(b->d_err);
    if (b->stream) cudaStreamDestroy(b->stream);
    delete b;
}

}  // namespace

extern "C" {

int it_batch_create(int32_t nsim, const it_sim_desc *descs, const it_params *common, it_batch **out) {
    if (!out) return bfail(IT_EINVAL, "out is NULL");
    *out = nullptr;
    if (nsim < 1 || !descs || !common) return bfail(IT_EINVAL, "need at least one simulation descriptor");
    if (common->precision != IT_FP32) return bfail(IT_EINVAL, "batched simulations use FP32 densities");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return bfail(IT_ECUDA, "no CUDA device available");
    it_batch *b = new (std::nothrow) it_batch();
    if (!b) return bfail(IT_ENOMEM, "host allocation failed");
    b->nsim = nsim;
    b->p = *common;
    b->desc.assign(descs, descs + nsim);
    b->hs.resize(nsim);
    b->dx.resize(nsim);
    b->dt.resize(nsim);
    b->steps.assign(nsim, 0);
    b->t_s.assign(nsim, 0.0);
    b->active.assign(nsim, 1);
    b->pulse_tracks.assign(nsim, {});
    b->pulse_count.assign(nsim, 1);
    b->pulse_done.assign(nsim, 0);
    b->pulse_period.assign(nsim, 0);
    b->chunk = 16384;
    b->cal[0] = b->cal[1] = b->cal[2] = 1.0;
    b->nmax.assign(nsim, 0.0);
    b->graph_parity = -1;
    size_t off = 0;
    for (int s = 0; s < nsim; ++s) {
        const it_sim_desc &d = descs[s];
        it_params p = *common;
        p.gap_cm = d.nz * d.dx_cm;
        p.voltage_V = d.voltage_V;
        p.n_peak_cm3 = d.n_peak_cm3;
        it_grid g{d.nx, d.ny, d.nz};
        double dt = d.dt_s;
        if (!(dt > 0)) {
            int rc = it_auto_dt(&p, d.dx_cm, &dt);
            if (rc) { batch_free(b); return rc; }
        }
        int rc = validate_step_args(&p, g, d.dx_cm, dt);
        if (rc) {
            std::string m = it_last_error();
            batch_free(b);
            return bfail(rc, "simulation " + std::to_string(s) + ": " + m);
        }
        if ((long long)d.nx * d.ny * d.nz > 0x7fffffffLL) {
            batch_free(b);
            return bfail(IT_EINVAL, "simulation " + std::to_string(s) + ": more than 2^31 - 1 cells");
        }
        BatchSim &h = b->hs[s];
        h.nx = d.nx; h.ny = d.ny; h.nz = d.nz; h.pad = 0;
        h.off = (long long)off;
        coef_f32(&p, d.dx_cm, dt, &h.cf);
        b->dx[s] = d.dx_cm;
        b->dt[s] = dt;
        const size_t cells = (size_t)d.nx * d.ny * d.nz;
        off += (cells + 63) / 64 * 64;   // 256-byte aligned per simulation
        b->max_nx = std::max(b->max_nx, d.nx);
        b->max_ny = std::max(b->max_ny, d.ny);
    }
    b->total = off;
    auto bail = [&](cudaError_t e, const char *what) {
        int rc = e == cudaErrorMemoryAllocation ? bfail(IT_ENOMEM, what) : cuda_fail(e, what);
        batch_free(b);
        return rc;
    };
    cudaError_t e;
    if ((e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking)) != cudaSuccess) return bail(e, "stream");
    if ((e = cudaMalloc(&b->state_base, sizeof(float) * 4 * off)) != cudaSuccess) return bail(e, "batch state");
    float *base = (float *)b->state_base;
    b->state[0][0] = base; b->state[0][1] = base + off; b->state[1][0] = base + 2 * off; b->state[1][1] = base + 3 * off;
    if ((e = cudaMemsetAsync(b->state_base, 0, sizeof(float) * 4 * off, b->stream)) != cudaSuccess) return bail(e, "memset");
    if ((e = cudaMalloc(&b->d_sims, sizeof(BatchSim) * nsim)) != cudaSuccess ||
        (e = cudaMalloc(&b->d_acc, sizeof(double) * NT * nsim)) != cudaSuccess ||
        (e = cudaMalloc(&b->d_rel, sizeof(double) * 8 * nsim)) != cudaSuccess ||
        (e = cudaMalloc(&b->d_tal, sizeof(double) * (NM * TAL_BLOCKS + TAL_OUT))) != cudaSuccess ||
        (e = cudaMalloc(&b->d_plane, sizeof(double) * 2 * b->max_nx * b->max_ny)) != cudaSuccess)   // plane + tile sums
        return bail(e, "batch scratch");
    if ((e = cudaMemcpyAsync(b->d_sims, b->hs.data(), sizeof(BatchSim) * nsim, cudaMemcpyHostToDevice, b->stream)) != cudaSuccess ||
        (e = cudaMemsetAsync(b->d_acc, 0, sizeof(double) * NT * nsim, b->stream)) != cudaSuccess ||
        (e = cudaMemsetAsync(b->d_rel, 0, sizeof(double) * 8 * nsim, b->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(b->stream)) != cudaSuccess)
        return bail(e, "batch setup");
    // tensor maps of the TMA batched kernel: simulations with nx % 4 == 0 and
    // nx <= 256 (one box spans the row); main boxes of min(256 / (nx/4), ny)
    // and min(512 / (nx/4), ny) rows (one or two float4 per thread) and a
    // box of one halo row
    b->tma_ok.assign(nsim, 0);
    {
        std::vector<CUtensorMap> maps((size_t)nsim * BT_MAPS);
        std::memset(maps.data(), 0, sizeof(CUtensorMap) * maps.size());
        for (int s = 0; s < nsim; ++s) {
            const BatchSim &h = b->hs[s];
            if (h.nx % 4 != 0 || h.nx > 256) continue;
            int rc = IT_OK;
            for (int set = 0; set < 2 && rc == IT_OK; ++set)
                for (int sp = 0; sp < 2 && rc == IT_OK; ++sp) {
                    float *base_s = b->state[set][sp] + h.off;
                    CUtensorMap *m = &maps[(size_t)s * BT_MAPS + set * 6 + sp * 3];
                    for (int ipt = 1; ipt <= 2 && rc == IT_OK; ++ipt)
                        rc = encode_map(&m[ipt - 1], base_s, h.nx, h.ny, h.nz, h.nx,
                                        std::min(tma_rows(h, ipt), h.ny));
                    if (rc == IT_OK) rc = encode_map(&m[2], base_s, h.nx, h.ny, h.nz, h.nx, 1);
                }
            if (rc) { batch_free(b); return rc; }
            b->tma_ok[s] = 1;
        }
        if ((e = cudaMalloc(&b->d_maps, sizeof(CUtensorMap) * maps.size())) != cudaSuccess ||
            (e = cudaMalloc(&b->d_err, sizeof(int))) != cudaSuccess ||
            (e = cudaMemcpyAsync(b->d_maps, maps.data(), sizeof(CUtensorMap) * maps.size(), cudaMemcpyHostToDevice,
                                 b->stream)) != cudaSuccess ||
            (e = cudaMemsetAsync(b->d_err, 0, sizeof(int), b->stream)) != cudaSuccess ||
            (e = cudaStreamSynchronize(b->stream)) != cudaSuccess)
            return bail(e, "batch tensor maps");
        for (auto *k : {step_batched_tma_kernel<true, true, 1>, step_batched_tma_kernel<true, false, 1>,
                        step_batched_tma_kernel<false, true, 1>, step_batched_tma_kernel<false, false, 1>})
            if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kBtSmem)) != cudaSuccess)
                return bail(e, "cudaFuncSetAttribute(batched TMA kernel)");
        for (auto *k : {step_batched_tma_kernel<true, true, 2>, step_batched_tma_kernel<true, false, 2>,
                        step_batched_tma_kernel<false, true, 2>, step_batched_tma_kernel<false, false, 2>})
            if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kBtSmem2)) != cudaSuccess)
                return bail(e, "cudaFuncSetAttribute(batched TMA kernel)");
    }
    b->tab_dirty = true;
    *out = b;
    return IT_OK;
}

}  // extern "C"

namespace {

// Deposit packed tracks [n][4] into simulation `sim`'s current set.  Nothing is
// waited for, so that the next simulation's deposit is prepared meanwhile: the
// host copy of pageable memory may run at any later time (a Grace host's pages
// need no staging), so packed points into the simulation's pulse_tracks, which
// outlive every copy.
int deposit_sim(it_batch *b, int sim, const double *packed, int64_t n) {
    if (n <= 0) return IT_OK;
    const it_sim_desc &d = b->desc[sim];
    const int parity = (int)(b->steps[sim] & 1);
    // a context view of this simulation for the shared deposition kernels
    it_ctx *v = new (std::nothrow) it_ctx();
    if (!v) return bfail(IT_ENOMEM, "host allocation failed");
    v->g = Grid{d.nx, d.ny, d.nz};
    v->dx = d.dx_cm;
    v->p = b->p;
    v->prec = IT_FP32;
    v->esize = 4;
    v->cur = 0;
    v->n[0][0] = b->state[parity][0] + b->hs[sim].off;
    v->n[0][1] = b->state[parity][1] + b->hs[sim].off;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    v->nmon = 2 * sms;
    v->d_plane = b->d_plane;
    v->d_acc = b->d_rel + (size_t)8 * sim;
    int rc = IT_OK;
    if (n > b->track_cap) {
        cudaFree(b->d_tracks); cudaFree(b->d_wx); cudaFree(b->d_wy);
        b->d_tracks = b->d_wx = b->d_wy = nullptr;
        b->track_cap = 0;
        cudaError_t e;
        if ((e = cudaMalloc(&b->d_tracks, kTrackScratch * n)) != cudaSuccess ||
            (e = cudaMalloc(&b->d_wx, sizeof(double) * b->max_nx * n)) != cudaSuccess ||
            (e = cudaMalloc(&b->d_wy, sizeof(double) * b->max_ny * n)) != cudaSuccess) {
            delete v;
            return cuda_fail(e, "batch track scratch");
        }
        b->track_cap = n;
    }
    cudaError_t e = cudaMemcpyAsync(b->d_tracks, packed, sizeof(double) * 4 * n, cudaMemcpyHostToDevice, b->stream);
    if (e != cudaSuccess) rc = cuda_fail(e, "track upload");
    v->d_tracks = b->d_tracks; v->d_wx = b->d_wx; v->d_wy = b->d_wy;
    if (rc == IT_OK) rc = launch_deposit(v, n, b->stream);
    delete v;
    return rc;
}

}  // namespace

extern "C" {

int it_batch_deposit_tracks(it_batch *b, int32_t sim, int64_t n, const double *xy, const double *let,
                            const double *bb) {
    if (!b || sim < 0 || sim >= b->nsim) return bfail(IT_EINVAL, "bad batch or simulation index");
    if (b->bstep != 0) return bfail(IT_ESTATE, "tracks are deposited before the first step");
    if (n < 0 || (n > 0 && (!xy || !let || !bb))) return bfail(IT_EINVAL, "bad track arrays");
    if (n == 0) return IT_OK;
    for (int64_t t = 0; t < n; ++t)
        if (!std::isfinite(xy[2 * t]) || !std::isfinite(xy[2 * t + 1]) || !(let[t] >= 0) || !std::isfinite(let[t]) ||
            !(bb[t] > 0) || !std::isfinite(bb[t]))
            return bfail(IT_EINVAL, "track values must be finite with LET >= 0 and b > 0");
    auto &pt = b->pulse_tracks[sim];
    // growing the simulation's list moves it: wait for the copies out of it
    if (!pt.empty()) IT_CK(cudaStreamSynchronize(b->stream));
    const size_t at = pt.size();
    pt.resize(at + (size_t)n * 4);
    double *packed = pt.data() + at;
    for (int64_t t = 0; t < n; ++t) {
        packed[4 * t] = xy[2 * t]; packed[4 * t + 1] = xy[2 * t + 1];
        packed[4 * t + 2] = let[t]; packed[4 * t + 3] = bb[t];
    }
    int rc = deposit_sim(b, sim, packed, n);
    if (rc) {
        cudaStreamSynchronize(b->stream);
        pt.resize(at);
        return rc;
    }
    b->pulse_done[sim] = 1;
    return IT_OK;
}

int it_batch_set_pulses(it_batch *b, int32_t sim, int32_t count, int64_t period_steps) {
    if (!b || sim < 0 || sim >= b->nsim) return bfail(IT_EINVAL, "bad batch or simulation index");
    if (b->bstep != 0) return bfail(IT_ESTATE, "pulse trains are set before the first step");
    if (count < 1 || (count > 1 && period_steps < 1)) return bfail(IT_EINVAL, "need count >= 1 and period_steps >= 1");
    b->pulse_count[sim] = count;
    b->pulse_period[sim] = period_steps;
    return IT_OK;
}

int it_batch_retime(it_batch *b) {
    if (!b) return bfail(IT_EINVAL, "batch is NULL");
    if (b->bstep != 0) return bfail(IT_ESTATE, "the time steps can only change before the first step");
    for (int s = 0; s < b->nsim; ++s) b->active[s] = 1;
    int rc = rebuild(b);
    if (rc) return rc;
    const int ne = (int)b->tab.size();
    float *d_mx = nullptr;
    IT_CK(cudaMalloc(&d_mx, sizeof(float) * ne));
    batch_max_kernel<<<ne, 256, 0, b->stream>>>(b->d_sims, b->d_tab, b->state[0][0], b->state[0][1], d_mx);
    cudaError_t e = cudaGetLastError();
    std::vector<float> mx(ne);
    if (e == cudaSuccess) e = cudaMemcpyAsync(mx.data(), d_mx, sizeof(float) * ne, cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    cudaFree(d_mx);
    if (e != cudaSuccess) return cuda_fail(e, "batch peak density");
    int a = -1;
    for (int s = 0; s < b->nsim; ++s) {
        ++a;   // every simulation is active here: a indexes mfirst/mcount
        if (b->desc[s].dt_s > 0) continue;
        double npk = 0.0;
        for (int q = b->mfirst[a]; q < b->mfirst[a] + b->mcount[a]; ++q) npk = std::max(npk, (double)mx[q]);
        npk *= std::max(1, b->pulse_count[s]);   // a train can pile its pulses up
        if (!std::isfinite(npk)) return bfail(IT_EUNSTABLE, "simulation " + std::to_string(s) + " is not finite");
        const it_sim_desc &d = b->desc[s];
        it_params p = b->p;
        p.gap_cm = d.nz * d.dx_cm;
        p.voltage_V = d.voltage_V;
        p.n_peak_cm3 = npk;
        double dt = 0.0;
        rc = it_auto_dt(&p, d.dx_cm, &dt);
        if (rc) return rc;
        b->dt[s] = dt;
        coef_f32(&p, d.dx_cm, dt, &b->hs[s].cf);
    }
    IT_CK(cudaMemcpyAsync(b->d_sims, b->hs.data(), sizeof(BatchSim) * b->nsim, cudaMemcpyHostToDevice, b->stream));
    IT_CK(cudaStreamSynchronize(b->stream));
    if (b->graph) { cudaGraphExecDestroy(b->graph); b->graph = nullptr; }
    return IT_OK;
}

int it_batch_set_chunk(it_batch *b, int64_t cells_per_block) {
    if (!b || cells_per_block < 256) return bfail(IT_EINVAL, "chunk must be at least 256 cells");
    b->chunk = cells_per_block;
    b->tab_dirty = true;
    return IT_OK;
}

int it_batch_autotune(it_batch *b, int32_t trial_steps, double *best_us) {
    if (!b) return bfail(IT_EINVAL, "batch is NULL");
    if (trial_steps < 2) return bfail(IT_EINVAL, "trial_steps must be at least 2");
    if (b->bstep != 0) return bfail(IT_ESTATE, "the launch shape is tuned before the first step");
    const int K = trial_steps + (trial_steps & 1);   // even: the state returns to set 0
    const size_t bytes = sizeof(float) * b->total;
    void *backup = nullptr;
    IT_CK(cudaMalloc(&backup, 2 * bytes));
    char *bk = (char *)backup;
    int rc = IT_OK;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaMemcpyAsync(bk, b->state[0][0], bytes, cudaMemcpyDeviceToDevice, b->stream) != cudaSuccess ||
        cudaMemcpyAsync(bk + bytes, b->state[0][1], bytes, cudaMemcpyDeviceToDevice, b->stream) != cudaSuccess ||
        cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        rc = cuda_fail(cudaGetLastError(), "batch autotune set-up");
    const long long chunk0 = b->chunk;
    // the entry size only shapes the single-cell march's entries: with no
    // simulation on it a single size is timed
    bool any_cells = false, any_tma = false;
    int active = 0;
    for (int s = 0; s < b->nsim; ++s)
        if (b->active[s]) {
            ++active;
            any_cells = any_cells || b->hs[s].nx % 4 != 0;
            any_tma = any_tma || b->tma_ok[s];
        }
    const std::vector<long long> chunks = any_cells ? std::vector<long long>{4096LL, 16384LL, 65536LL}
                                                    : std::vector<long long>{chunk0};
    // candidates: the TMA kernels with z splits aiming at 1..32 CTAs per SM,
    // each distinct split once; the direct march with the fitted chunk of
    // planes and half of it
    const int sms = sm_count();
    std::vector<BatchShape> shapes;
    if (any_tma)
        for (int tma : {2, 1}) {
            int seen = 0;
            for (int cps : {1, 2, 4, 8, 16, 32}) {
                const BatchShape sh{tma, cps};
                const int split = tma_split(b, sh, sms);
                if (split != seen) shapes.push_back(sh);
                seen = split;
            }
        }
    shapes.push_back({0, 1});
    shapes.push_back({0, 2});
    long long best_chunk = chunk0;
    BatchShape best_shape = b->shape;
    double best = 1e300, kind_us[3] = {1e300, 1e300, 1e300}, kind_fit[3] = {0.0, 0.0, 0.0};
    for (const BatchShape &sh : shapes)
        for (long long chunk : chunks) {
            if (rc) break;
            b->shape = sh;
            b->chunk = chunk;
            rc = build_table(b);
            // two steps show a candidate that is out of the running (slower
            // than the best by more than a twentieth); the others are timed
            int done = 0;
            double us = 0.0;
            for (const int want : {std::min(2, K), K}) {
                float ms = 0.f;
                for (int q = 0; q < (done ? 0 : 2) && !rc; ++q) rc = launch_batched_step(b, q & 1);
                const int n = want;
                if (!rc && cudaEventRecord(e0, b->stream) != cudaSuccess) rc = cuda_fail(cudaGetLastError(), "event");
                for (int q = 0; q < n && !rc; ++q) rc = launch_batched_step(b, q & 1);
                if (!rc && cudaEventRecord(e1, b->stream) != cudaSuccess) rc = cuda_fail(cudaGetLastError(), "event");
                if (!rc) {
                    cudaError_t e = cudaEventSynchronize(e1);
                    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                    if (e != cudaSuccess) rc = cuda_fail(e, "batch autotune timing");
                }
                us = ms * 1e3 / n;
                done += n;
                if (rc || done >= K || us > 1.05 * best) break;
            }
            // the trial steps changed the state: put the deposited state back
            if (cudaMemcpyAsync(b->state[0][0], bk, bytes, cudaMemcpyDeviceToDevice, b->stream) != cudaSuccess ||
                cudaMemcpyAsync(b->state[0][1], bk + bytes, bytes, cudaMemcpyDeviceToDevice, b->stream) != cudaSuccess)
                rc = rc ? rc : cuda_fail(cudaGetLastError(), "batch autotune restore");
            if (rc) break;
            if (us < kind_us[sh.tma]) {
                kind_us[sh.tma] = us;
                kind_fit[sh.tma] = shape_us(b, sh, sms);
            }
            if (done >= K && us < best) {
                best = us;
                best_chunk = chunk;
                best_shape = sh;
            }
        }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaStreamSynchronize(b->stream);
    cudaFree(backup);
    // the chosen shape; the next table build also clears the trial tallies
    b->chunk = rc ? chunk0 : best_chunk;
    if (!rc) {
        b->tuned = true;
        b->tuned_shape = best_shape;
        b->tuned_active = active;
        // the fit's error at full occupancy scales it as simulations finish
        for (int k = 0; k < 3; ++k)
            if (kind_fit[k] > 0.0) b->cal[k] = kind_us[k] / kind_fit[k];
    }
    b->tab_dirty = true;
    if (b->graph) { cudaGraphExecDestroy(b->graph); b->graph = nullptr; }
    if (rc) return rc;
    if (best_us) *best_us = best;
    return IT_OK;
}

int it_batch_get_launch(it_batch *b, int *float4_per_thread, int *ctas_per_sm) {
    if (!b) return bfail(IT_EINVAL, "batch is NULL");
    const BatchShape sh = choose_shape(b, sm_count());
    if (float4_per_thread) *float4_per_thread = sh.tma;
    if (ctas_per_sm) *ctas_per_sm = sh.tma ? sh.cps : 0;
    return IT_OK;
}

int it_test_batch_launch(it_batch *b, int float4_per_thread, int ctas_per_sm) {
    if (!b) return bfail(IT_EINVAL, "batch is NULL");
    if (float4_per_thread < -1 || float4_per_thread > 2 || (float4_per_thread >= 0 && (ctas_per_sm < 1 || ctas_per_sm > 64)))
        return bfail(IT_EINVAL, "0 to 2 float4 per thread and 1 to 64 CTAs per SM (-1: the choice is free)");
    b->forced = float4_per_thread >= 0;
    if (b->forced) b->forced_shape = BatchShape{float4_per_thread, ctas_per_sm};
    b->tab_dirty = true;
    return IT_OK;
}

int it_batch_run(it_batch *b, double tol, int64_t max_steps, int64_t check_every, int64_t *launches) {
    if (!b) return bfail(IT_EINVAL, "batch is NULL");
    if (!(tol >= 0) || max_steps < 0 || check_every < 2) return bfail(IT_EINVAL, "bad argument");
    const int K = (int)(check_every + (check_every & 1));
    for (int s = 0; s < b->nsim; ++s)
        if (b->pulse_count[s] > 1 && b->pulse_period[s] % K != 0)
            return bfail(IT_EINVAL, "simulation " + std::to_string(s) + ": pulse period must be a multiple of the even check interval");
    std::vector<double> rel(8 * (size_t)b->nsim);
    IT_CK(cudaMemcpyAsync(rel.data(), b->d_rel, sizeof(double) * 8 * b->nsim, cudaMemcpyDeviceToHost, b->stream));
    IT_CK(cudaStreamSynchronize(b->stream));
    int64_t nl = 0;
    std::vector<double> ind;
    for (;;) {
        if (b->tab_dirty) {
            int rc = rebuild(b);
            if (rc) return rc;
        }
        // next pulse of a train: deposited at the start of its step
        bool deposited = false;
        for (size_t a = 0; a < b->sim_of.size(); ++a) {
            const int s = b->sim_of[a];
            const int done = b->pulse_done[s];
            if (done >= 1 && done < b->pulse_count[s] && b->steps[s] == (int64_t)done * b->pulse_period[s]) {
                const auto &pt = b->pulse_tracks[s];
                int rc = deposit_sim(b, s, pt.data(), (int64_t)(pt.size() / 4));
                if (rc) return rc;
                b->pulse_done[s] = done + 1;
                deposited = true;
            }
        }
        if (deposited) {
            IT_CK(cudaMemcpyAsync(rel.data(), b->d_rel, sizeof(double) * 8 * b->nsim, cudaMemcpyDeviceToHost, b->stream));
            IT_CK(cudaStreamSynchronize(b->stream));
        }
        // completion of every active simulation
        int rc = in_domain(b, ind);
        if (rc) return rc;
        bool changed = false;
        for (size_t a = 0; a < b->sim_of.size(); ++a) {
            const int s = b->sim_of[a];
            const double r = rel[8 * s] + rel[8 * s + 1];
            const double in = ind[2 * s] + ind[2 * s + 1];
            if (!std::isfinite(in)) return bfail(IT_EUNSTABLE, "simulation " + std::to_string(s) + " is not finite");
            const bool pending = b->pulse_done[s] >= 1 && b->pulse_done[s] < b->pulse_count[s];
            if (r <= 0 || (!pending && in / r < tol) || b->steps[s] >= max_steps) {
                b->active[s] = 0;
                changed = true;
            }
        }
        if (changed) {
            rc = rebuild(b);
            if (rc) return rc;
        }
        if (b->tab.empty()) break;
        if (b->p.dt_ladder) {
            rc = ladder_batch(b);
            if (rc) return rc;
        }
        rc = run_segment(b, K);
        if (rc) return rc;
        nl += K;
        rc = fold(b);
        if (rc) return rc;
    }
    if (launches) *launches = nl;
    IT_CK(cudaStreamSynchronize(b->stream));
    return IT_OK;
}

int it_batch_tallies(it_batch *b, int32_t sim, it_tallies_t *t) {
    if (!b || !t || sim < 0 || sim >= b->nsim) return bfail(IT_EINVAL, "bad argument");
    // in-domain charge and extreme densities of this simulation's current set,
    // then everything in one copy
    const size_t cells = (size_t)b->hs[sim].nx * b->hs[sim].ny * b->hs[sim].nz;
    const int parity = (int)(b->steps[sim] & 1);
    const double vol = b->dx[sim] * b->dx[sim] * b->dx[sim];
    double *d_out = b->d_tal + NM * TAL_BLOCKS;
    int rc = launch_monitor_raw_f32(b->state[parity][0] + b->hs[sim].off, b->state[parity][1] + b->hs[sim].off,
                                    cells, vol, b->d_tal, TAL_BLOCKS, b->stream);
    if (rc) return rc;
    batch_tally_kernel<<<1, TAL_OUT * 32, 0, b->stream>>>(b->d_acc + (size_t)NT * sim, b->d_rel + (size_t)8 * sim,
                                                          b->d_tal, d_out);
    IT_CK(cudaGetLastError());
    double o[TAL_OUT];
    IT_CK(cudaMemcpyAsync(o, d_out, sizeof(o), cudaMemcpyDeviceToHost, b->stream));
    IT_CK(cudaStreamSynchronize(b->stream));
    std::memset(t, 0, sizeof(*t));
    const double *rel = o + NT;
    for (int s = 0; s < 2; ++s) {
        t->released[s] = rel[s];
        t->in_domain[s] = o[NT + 2 + s];
        t->n_min[s] = o[NT + 4 + s];
        t->n_max[s] = o[NT + 6 + s];
    }
    t->recombined = o[0];
    t->collected_anode[0] = o[1]; t->collected_anode[1] = o[2];
    t->collected_cathode[0] = o[3]; t->collected_cathode[1] = o[4];
    t->lost_lateral[0] = o[5]; t->lost_lateral[1] = o[6];
    t->space_charge[0] = o[7]; t->space_charge[1] = o[8];
    const double r = rel[0] + rel[1];
    t->f = r > 0 ? (o[1] + o[2] + o[3] + o[4]) / r : NAN;
    t->steps = b->steps[sim];
    t->dt_s = b->dt[sim];
    t->t_s = b->t_s[sim];
    return IT_OK;
}

int it_batch_get_density(it_batch *b, int32_t sim, int species, void *dst, size_t bytes) {
    if (!b || !dst || sim < 0 || sim >= b->nsim || (species != 0 && species != 1)) return bfail(IT_EINVAL, "bad argument");
    const size_t cells = (size_t)b->hs[sim].nx * b->hs[sim].ny * b->hs[sim].nz;
    if (bytes != cells * sizeof(float)) return bfail(IT_EINVAL, "bytes must equal cells * 4");
    const int parity = (int)(b->steps[sim] & 1);
    IT_CK(cudaMemcpyAsync(dst, b->state[parity][species] + b->hs[sim].off, bytes, cudaMemcpyDeviceToHost, b->stream));
    IT_CK(cudaStreamSynchronize(b->stream));
    return IT_OK;
}

int it_batch_destroy(it_batch *b) {
    batch_free(b);
    return IT_OK;
}

}  // extern "C"
