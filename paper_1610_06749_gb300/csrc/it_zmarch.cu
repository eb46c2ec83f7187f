// it_zmarch.cu -- launch shapes and tensor maps of the staged march
// (it_zmarch.cuh), and its instances with plain sums.
#include <cudaTypedefs.h>

#include <cstdlib>

#include "it_zmarch.cuh"

namespace itk {

template cudaError_t zm_prepare_shape<false>(bool, int, int, bool, bool, size_t, int *);
template void zm_launch_shape<false>(bool, int, int, bool, bool, int, const ZmMaps &, const float *, const float *,
                                    float *, float *, int, int, int,
                                    const ZmConf &, const Coef<float> &, double *, int *, cudaStream_t);

// ---------------------------------------------------------------------------
// host side: launch shape and tensor maps
// ---------------------------------------------------------------------------
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

int encode_map(CUtensorMap *m, void *base, int nx, int ny, int nz, int bx, int rows) {
    auto fn = encode_fn();
    if (!fn) {
        set_error("cuTensorMapEncodeTiled is not available");
        return IT_ECUDA;
    }
    cuuint64_t dims[3] = {(cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)nz};
    cuuint64_t strides[2] = {(cuuint64_t)nx * 4, (cuuint64_t)nx * ny * 4};
    cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (code " + std::to_string((int)r) + ")");
        return IT_ECUDA;
    }
    return IT_OK;
}

// Width of the pieces a row of nx > 256 floats is split into: its largest
// divisor that is a multiple of 4 floats (16-byte strides) and fits a box
// dimension (256).  0: no divisor of at least 128 bytes, whose boxes would
// crawl in 16-byte pieces, or too many pieces for a box dimension.
int row_piece(int nx) {
    for (int d = 256; d >= 32; d -= 4)
        if (nx % d == 0) return nx / d <= 256 ? d : 0;
    return 0;
}

// Wide rows (nx > 256): a 4-D view {d, nx / d, ny, nz} of the same array with
// d = row_piece(nx) (byte strides of a piece, a row, a plane), boxes of
// {d, nx / d, rows, 1}, which land in shared memory as `rows` whole rows of
// nx floats: one copy per box where the 3-D view needs nx / d.
int encode_map_rows(CUtensorMap *m, void *base, int nx, int ny, int nz, int rows) {
    auto fn = encode_fn();
    if (!fn) {
        set_error("cuTensorMapEncodeTiled is not available");
        return IT_ECUDA;
    }
    const int d = row_piece(nx), xs = nx / d;
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)xs, (cuuint64_t)ny, (cuuint64_t)nz};
    cuuint64_t strides[3] = {(cuuint64_t)d * 4, (cuuint64_t)nx * 4, (cuuint64_t)nx * ny * 4};
    cuuint32_t box[4] = {(cuuint32_t)d, (cuuint32_t)xs, (cuuint32_t)rows, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled (row view) failed (code " + std::to_string((int)r) + ")");
        return IT_ECUDA;
    }
    return IT_OK;
}

// bf16 operand of the tensor-core GEMM (it_tc.cuh): dims {K, rows, members}
// (K contiguous), byte strides of a row and of a member, boxes of 64 x
// box_rows with the 128-byte swizzle; rows and K beyond the dims arrive as zeros.
int encode_bf16_sw128(CUtensorMap *m, const void *base, long long K, long long rows, long long members,
                      long long row_bytes, long long member_bytes, int box_rows) {
    auto fn = encode_fn();
    if (!fn) {
        set_error("cuTensorMapEncodeTiled is not available");
        return IT_ECUDA;
    }
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)members};
    cuuint64_t strides[2] = {(cuuint64_t)row_bytes, (cuuint64_t)member_bytes};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled (bf16 operand) failed (code " + std::to_string((int)r) + ")");
        return IT_ECUDA;
    }
    return IT_OK;
}

static int align32f(int floats) { return (floats + 31) / 32 * 32; }   // 128-byte multiple of floats

static int ipt_of(const it_ctx *c, int TY, int nw) { return ((c->g.nx / 4) * TY + nw * 32 - 1) / (nw * 32); }

static int sm_count() {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// A thread's two (four) items as vertically adjacent rows?
static bool zm_pairs(const it_ctx *c, int TY, int nw) {
    const int ipt = ipt_of(c, TY, nw);
    return ipt % 2 == 0 && TY % 2 == 0 && (c->g.nx / 4) * (TY / 2) <= (ipt / 2) * nw * 32;
}

// Tile height, CTAs per SM and grid when none is given: the shape with the
// least fitted time, returned in us.  A CTA takes (planes it walks + 2) rounds
// and about 4 us to start and drain.  A round is bound by memory or by the
// CTA's own chain of wait, update and hand-over:
//   * memory: 16 bytes per cell of all CTAs at 6.5 TB/s (2.46 ps per cell),
//     times 1 + 0.75 / TY^2 when the grid is a multiple of the tile count (all
//     tile columns are then cut at the same z and adjacent tiles stream in
//     step, so that their halo rows come from L2), else 1 + 1 / TY (the two
//     halo rows come from HBM);
//   * the chain: 0.82 and 1.25 us with one and two float4 per thread and a
//     producer, 1.7 / 2.0 / 3.2 for two to four without, 1.25 / 1.62 / 2.4 /
//     4.3 with space charge; 10 % more at one CTA per SM without a producer,
//     5 % more where the halo rows come from HBM.
// Fitted to launch-shape sweeps on 18 grids, where the choice is the fastest
// shape or within 3 % of it on all but four (within 10 %): 256x256x400 8 rows,
// 2 CTAs per SM: 70 us (16 rows, 1 CTA: 72); 512x512x256 8 rows, 1 CTA: 170
// (the whole 304 slots instead of a multiple of the tile count: 238);
// 768x768x100 8 rows, 1 CTA, all 152 slots: 174 (4 rows, 2 CTAs: 207);
// 1024x256x200 4 rows, 1 CTA: 138 (2 rows, 2 CTAs: 151); 384x320x128 with
// space charge 8 rows, 2 CTAs: 53 (5 rows, 2 CTAs: 59).
static double zmarch_shape(const it_ctx *c, int *ty, int *cps, long long *ctas) {
    static const double prod_us[2] = {0.82, 1.25}, ring_us[4] = {1.25, 1.7, 2.0, 3.2}, sc_us[4] = {1.25, 1.62, 2.4, 4.3};
    const int sms = sm_count();
    const bool sc = c->p.space_charge != 0, per = c->p.lateral_bc == IT_PERIODIC;
    double best = 1e300;
    for (int k = 2; k >= 1; --k)
        for (int t = 1; t <= std::min(c->g.ny, 255); ++t) {
            if (c->g.ny % t) continue;
            const int nw = k == 1 ? 16 : 8, ipt = ipt_of(c, t, nw);
            if (ipt > ZM_MAX_IPT) break;
            const size_t slot = sizeof(float) * 2 * (align32f(t * c->g.nx) + 2 * align32f(c->g.nx));
            if (3 * slot + 512 > (size_t)(220 * 1024) / k) continue;   // a ring of three slots must fit
            const int ntile = c->g.ny / t;
            const long long tp = (long long)ntile * c->g.nz, slots = (long long)sms * k;
            const double chain = zm_prod(per, ipt, sc, zm_pairs(c, t, nw))
                                     ? prod_us[ipt - 1]
                                     : (sc ? sc_us : ring_us)[ipt - 1] * (k == 1 ? 1.1 : 1.0);
            for (int aligned = 1; aligned >= 0; --aligned) {
                if (aligned && slots < ntile) continue;
                const long long grid = std::min(tp, aligned ? slots / ntile * ntile : slots);
                const double mem = 2.46e-6 * (double)(grid * t * c->g.nx) * (1.0 + (aligned ? 0.75 / t : 1.0) / t);
                const double us = (double)((tp + grid - 1) / grid + 2) * std::max(aligned ? chain : 1.05 * chain, mem) + 4.0;
                if (us < 0.98 * best) {
                    best = us;
                    *ty = t;
                    *cps = k;
                    *ctas = grid;
                }
            }
        }
    return best;
}

// Fill c->zm for a requested tile height / CTAs per SM / ring depth
// (0 = choose) and build the tensor maps.  One CTA per SM runs 16 warps,
// two CTAs per SM run 8 warps each.
int zmarch_setup(it_ctx *c, int want_ty, int want_cps, int want_s, int want_grid) {
    const int nx = c->g.nx, ny = c->g.ny, nz = c->g.nz;
    if (c->prec != IT_FP32) { set_error("z-march kernel needs FP32 densities"); return IT_EINVAL; }
    if (nx % 4 != 0) { set_error("z-march kernel needs nx % 4 == 0"); return IT_EINVAL; }
    if (nx > 256 && !row_piece(nx)) {
        set_error("z-march kernel: nx > 256 needs a divisor of 32 to 256 that is a multiple of 4");
        return IT_EINVAL;
    }
    if ((unsigned long long)nx * ny * nz > 0xFFFFFFFFull) {
        set_error("z-march kernel indexes a species array with 32 bits: needs nx*ny*nz < 2^32");
        return IT_EINVAL;
    }
    int cps = want_cps > 0 ? want_cps : 1, TY = want_ty;
    long long ctas = 0;
    if (want_ty <= 0 && want_cps <= 0) zmarch_shape(c, &TY, &cps, &ctas);
    if (cps > 2) { set_error("z-march kernel runs 1 or 2 CTAs per SM"); return IT_EINVAL; }
    const int nw = cps == 1 ? 16 : 8;
    ZmConf z{};
    z.threads = nw * 32;
    // a ring block holds whole rows; rows wider than a TMA box dimension (256
    // floats) come through the 4-D view (one box of several pieces per row)
    z.xs = nx > 256 ? nx / row_piece(nx) : 1;
    z.bx = nx;
    z.nbx = 1;
    // CTAs per SM given: the smallest divisor of ny that gives every thread
    // two float4 items (else the largest with at most ZM_MAX_IPT)
    if (TY <= 0) {
        TY = 0;
        for (int t = 1; t <= ny; ++t) {
            if (ny % t) continue;
            if (ipt_of(c, t, nw) > ZM_MAX_IPT) break;
            TY = t;
            if ((nx / 4) * t >= 2 * z.threads) break;
        }
    }
    if (TY <= 0 || ny % TY != 0 || ipt_of(c, TY, nw) > ZM_MAX_IPT || TY > 255) {
        set_error("z-march kernel: no usable tile height for this grid");
        return IT_EINVAL;
    }
    z.TY = TY;
    z.ntile = ny / TY;
    z.reg_top = 0;
    z.reg_main = align32f(z.bx);
    z.reg_bot = z.reg_main + align32f(TY * z.bx);
    z.blk = z.reg_bot + align32f(z.bx);
    z.slot = 2 * z.nbx * z.blk;
    const size_t budget = (size_t)(220 * 1024) / cps;
    const bool per = c->p.lateral_bc == IT_PERIODIC;
    const int ipt = ipt_of(c, TY, nw);
    const bool sc = c->p.space_charge != 0, exact = exact_sums(nx);
    z.pair = zm_pairs(c, TY, nw);
    // ring depth: with a producer the smallest (of 4 and more) that keeps
    // 64 KB per SM in flight beyond the two planes in use; deeper rings only
    // spread the CTAs' planes (256x256x400, 8 rows, 2 CTAs per SM: 71.6 / 69.8
    // / 76.6 us with 3 / 4 / 5 slots; 200x200x800 absorbing, 10 rows: 85.2 /
    // 90.5 with 4 / 5).  Otherwise what fits, up to 8.
    z.S = want_s > 0 ? want_s : 8;
    if (want_s <= 0 && zm_prod(per, ipt, sc, z.pair))
        for (z.S = 4; z.S < 8 && (size_t)(z.S - 2) * z.slot * sizeof(float) * cps < 64 * 1024;) ++z.S;
    if (z.S < 3 || z.S > 16) { set_error("z-march ring depth must be 3..16"); return IT_EINVAL; }
    for (;;) {
        z.smem = (size_t)z.S * z.slot * sizeof(float) + 16 * z.S + 128;   // ring + barriers (and counters) + alignment slack
        if (z.smem <= budget || z.S == 3 || want_s > 0) break;
        --z.S;
    }
    if (z.smem > 227 * 1024) { set_error("z-march kernel: tile does not fit in shared memory"); return IT_EINVAL; }
    int occ = cps;
    cudaError_t e = exact ? zm_prepare_shape<true>(per, ipt, nw, sc, z.pair, z.smem, &occ)
                          : zm_prepare_shape<false>(per, ipt, nw, sc, z.pair, z.smem, &occ);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(z-march)");
    if (occ < cps) { set_error("z-march kernel: requested CTAs per SM do not fit"); return IT_EINVAL; }
    z.ctas_per_sm = cps;
    const int sms = sm_count();
    // grid: CTAs, each taking one contiguous range of tile-planes.  0: one
    // per resident slot (with no shape given at all, zmarch_shape's choice);
    // -1: the largest multiple of the tile count that fits the resident slots,
    // so every tile column is cut at the same z and vertically adjacent tiles
    // are streamed in step (their halo rows are then still in L2); > 0: as
    // given.
    const long long tp = (long long)z.ntile * nz;
    long long grid = (long long)sms * cps;
    if (want_grid == -1 && grid >= z.ntile) grid = grid / z.ntile * z.ntile;
    else if (want_grid > 0) grid = want_grid;
    else if (want_s <= 0 && ctas > 0) grid = ctas;
    z.nzc = (int)std::min<long long>(grid, tp);
    for (int set = 0; set < 2; ++set)
        for (int s = 0; s < 2; ++s) {
            int rc = z.xs > 1 ? encode_map_rows(&c->tm_main[set][s], c->n[set][s], nx, ny, nz, TY)
                              : encode_map(&c->tm_main[set][s], c->n[set][s], nx, ny, nz, z.bx, TY);
            if (rc) return rc;
            rc = z.xs > 1 ? encode_map_rows(&c->tm_halo[set][s], c->n[set][s], nx, ny, nz, 1)
                          : encode_map(&c->tm_halo[set][s], c->n[set][s], nx, ny, nz, z.bx, 1);
            if (rc) return rc;
        }
    c->zm = z;
    c->zm_grid = z.nzc;
    return IT_OK;
}

// Does the march straight from L1/L2 (step_direct_kernel) beat the TMA-staged
// one?  By the fitted times of both: it does while the state stays in L2
// (128x128x200: 12.4 against 19.6 us per step, 256x256x100: 22.8 against a
// fitted 24.6) and where ny has no divisor that fills a tile (224x293x119: one
// row per tile took 154 us); from HBM it moves 1.45 times slower than a copy
// and the ring wins (256x256x400: 86 against 70).
bool direct_wins(const it_ctx *c) {
    int ty = 0, cps = 1;
    long long ctas = 0;
    return direct_us(c) < zmarch_shape(c, &ty, &cps, &ctas);
}

int zmarch_configure(it_ctx *c) { return zmarch_setup(c, 0, 0, 0, 0); }

int launch_step_zmarch(it_ctx *c, cudaStream_t s) {
    if (c->direct) return launch_step_direct(c, s);
    const int cur = c->cur, nxt = cur ^ 1;
    ZmMaps maps;
    maps.main[0] = c->tm_main[cur][0];
    maps.main[1] = c->tm_main[cur][1];
    maps.halo[0] = c->tm_halo[cur][0];
    maps.halo[1] = c->tm_halo[cur][1];
    const float *ip = (const float *)c->n[cur][0], *im = (const float *)c->n[cur][1];
    float *op = (float *)c->n[nxt][0], *om = (float *)c->n[nxt][1];
    ZmConf z = c->zm;
    z.wait_cycles = c->wait_cycles > 0 ? c->wait_cycles : (1LL << 32);
    z.withhold = c->withhold;
    const bool per = c->p.lateral_bc == IT_PERIODIC;
    const int nw = z.threads / 32;
    const int ipt = ipt_of(c, z.TY, nw);
    const int nx = c->g.nx, ny = c->g.ny, nz = c->g.nz;
    const bool sc = c->p.space_charge != 0, exact = exact_sums(nx);
    const bool down = cur != c->base;   // alternate steps, alternate directions
    auto *launch = exact ? zm_launch_shape<true> : zm_launch_shape<false>;
    launch(per, ipt, nw, sc, down, c->zm_grid, maps, ip, im, op, om, nx, ny, nz, z, c->cf, c->d_slots, c->d_err, s);
    IT_CK(cudaGetLastError());
    c->cur = nxt;
    return IT_OK;
}

}  // namespace itk
