// it_mlp.cu -- the surrogate network for the collection efficiency f.
//
// A 6 -> 256 -> 256 -> 256 -> 256 -> 1 perceptron with SiLU hidden layers
// and a sigmoid output, an ensemble of independent members trained on
// solver results.  Weights are stored in bfloat16 for the matrix products
// (FP32 master copies for Adam), all products accumulate in FP32 on the
// tensor cores, bias, SiLU and its derivative are fused into the product
// epilogues, and the output layer, sigmoid, squared error and the first
// backward step are one fused kernel.  Every reduction runs in a fixed order
// (bitwise-reproducible training).
//
// Precision: weights enter the products as bf16; each layer's input enters
// as a two-term bf16 expansion hi + lo (hi = bf16(a), lo = bf16(a - hi),
// about 16 significant bits) against the weights duplicated along K, so the
// forward pass carries bf16 weights but near-FP32 activations.  A
// one-term bf16 activation added rounding noise of ~2e-4 to f on held-out
// configurations (median; FP64 activations with the same weights: ~1e-4).
// Error signals and the activations of the weight gradients stay one-term
// bf16.
//
// The 256 x 256 products (forward of layers 2-4, their data gradients and
// weight gradients) run on the 5th-generation tensor cores (it_tc.cuh:
// TMA-staged bf16 tiles, tcgen05.mma into tensor memory, fused epilogues).
// Both operands are K-major, so the data gradient reads transposed weight
// copies and the weight gradient reads transposed activations and error
// signals, which the producing epilogues write beside the row-major ones.
// The first layer (6 inputs) and its weight gradient are too narrow for
// them and take one small mma.sync product per warp.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "it_device.cuh"
#include "it_internal.cuh"
#include "it_tc.cuh"

namespace itk {
namespace mlp {

constexpr int H = IT_MLP_HIDDEN;
constexpr int NIN = IT_MLP_INPUTS;
// parameter offsets inside one member (W stored out x in)
constexpr long long OW1 = 0, OB1 = OW1 + (long long)H * NIN, OW2 = OB1 + H, OB2 = OW2 + (long long)H * H,
                    OW3 = OB2 + H, OB3 = OW3 + (long long)H * H, OW4 = OB3 + H, OB4 = OW4 + (long long)H * H,
                    OW5 = OB4 + H, OB5 = OW5 + H, P = OB5 + 1;
static_assert(P == IT_MLP_PARAMS, "parameter layout");

__device__ __forceinline__ float silu(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float dsilu(float z) {
    const float s = 1.f / (1.f + __expf(-z));
    return s * (1.f + z * (1.f - s));
}

// One 16 x 8 x 16 product on mma.sync (bf16 operands, FP32 accumulation).
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Output layer, sigmoid, squared error and the first backward step, one warp
// per (sample, member), eight samples per block: z = A4 . w5 + b5, fhat =
// sigmoid(z); when training, dz = 2/B (fhat - y) fhat (1 - fhat), dZ4 = dz w5 *
// SiLU'(Z4) (fp32, bf16 and bf16 transposed, whose eight samples of a row are
// written together).
__global__ void __launch_bounds__(256)
out_layer_kernel(const __nv_bfloat16 *__restrict__ A4, const float *__restrict__ Z4,
                 const __nv_bfloat16 *__restrict__ w, const float *__restrict__ master,
                 const float *__restrict__ y, long long ybs, int B, int train, float *__restrict__ fhat,
                 float *__restrict__ dzout, float *__restrict__ dZ, __nv_bfloat16 *__restrict__ dZb,
                 long long zact, __nv_bfloat16 *__restrict__ dZbT, long long zT, long long ldT, long long zA) {
    __shared__ __align__(16) __nv_bfloat16 tile[H][8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * 8, m = m0 + warp;
    const int z = blockIdx.y;
    if (m < B) {
        const __nv_bfloat16 *w5 = w + z * P + OW5;
        const __nv_bfloat16 *a = A4 + z * zA + (long long)m * 2 * H;   // hi | lo
        float wk[H / 32], zk[H / 32];
        const long long o = z * zact + (long long)m * H + lane;
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < H / 32; ++q) {
            const int k = lane + 32 * q;
            wk[q] = __bfloat162float(w5[k]);
            zk[q] = train ? Z4[o + 32 * q] : 0.f;
            s += (__bfloat162float(a[k]) + __bfloat162float(a[k + H])) * wk[q];
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        const float zz = s + master[z * P + OB5];
        const float f = 1.f / (1.f + __expf(-zz));
        if (lane == 0) fhat[z * B + m] = f;
        if (train) {
            const float dz = 2.f / B * (f - y[(long long)z * ybs + m]) * f * (1.f - f);
            if (lane == 0) dzout[z * B + m] = dz;
#pragma unroll
            for (int q = 0; q < H / 32; ++q) {
                const float d = dz * wk[q] * dsilu(zk[q]);
                dZ[o + 32 * q] = d;
                const __nv_bfloat16 db = __float2bfloat16_rn(d);
                dZb[o + 32 * q] = db;
                tile[lane + 32 * q][warp] = db;
            }
        }
    }
    if (!train) return;
    __syncthreads();
    __nv_bfloat16 *dst = dZbT + z * zT + (long long)threadIdx.x * ldT + m0;
    if (m0 + 8 <= B) {
        *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(&tile[threadIdx.x][0]);
    } else {
        for (int r = 0; r < B - m0; ++r) dst[r] = tile[threadIdx.x][r];
    }
}

// grad of w5 and b5 (fixed order over the batch): g[k] = sum_m dz[m] A4[m][k]
// (A4 = hi + lo, as in the forward pass).
// Block (x, member), 8 warps: lane c of warp w sums column k = 32 x + c over
// the rows m = w, w + 8, ...; the 8 partial sums are added in warp order.
// Block x = 0 also forms b5's sum (thread t over m = t, t + 256, ..., then
// the 256 partials in thread order).
__global__ void __launch_bounds__(256)
out_grad_kernel(const __nv_bfloat16 *__restrict__ A4, const float *__restrict__ dz, int B, float *__restrict__ grad,
                long long zA) {
    __shared__ float part[8][33];
    __shared__ float bpart[256];
    const int z = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    const __nv_bfloat16 *a = A4 + z * zA;   // rows of hi | lo
    const float *d = dz + (long long)z * B;
    float s = 0.f;
    for (int m = warp; m < B; m += 8)
        s += d[m] * (__bfloat162float(a[(long long)m * 2 * H + k]) + __bfloat162float(a[(long long)m * 2 * H + H + k]));
    part[warp][lane] = s;
    if (blockIdx.x == 0) {
        float t = 0.f;
        for (int m = threadIdx.x; m < B; m += 256) t += d[m];
        bpart[threadIdx.x] = t;
    }
    __syncthreads();
    if (warp == 0) {
        float g = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) g += part[w][lane];
        grad[z * P + OW5 + k] = g;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        float t = 0.f;
        for (int q = 0; q < 256; ++q) t += bpart[q];
        grad[z * P + OB5] = t;
    }
}

// bias gradient: column sums of dZ [B][H], fixed order.  Block (x, member),
// 8 warps: lane c of warp w sums column n = 32 x + c over the rows m = w,
// w + 8, ...; the 8 partial sums are added in warp order.
__global__ void __launch_bounds__(256)
bias_grad_kernel(const float *__restrict__ dZ, int B, float *__restrict__ grad, long long off, long long zact) {
    __shared__ float part[8][33];
    const int z = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = blockIdx.x * 32 + lane;
    const float *d = dZ + z * zact;
    float s = 0.f;
    for (int m = warp; m < B; m += 8) s += d[(long long)m * H + n];
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        float g = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) g += part[w][lane];
        grad[z * P + off + n] = g;
    }
}

// mean squared error per member, fixed order
__global__ void loss_kernel(const float *__restrict__ fhat, const float *__restrict__ y, long long ybs, int B,
                            double *__restrict__ loss, int accumulate) {
    __shared__ double red[32];
    const int z = blockIdx.x;
    double v[1] = {0.0};
    for (int m = threadIdx.x; m < B; m += blockDim.x) {
        const double d = (double)fhat[z * B + m] - (double)y[(long long)z * ybs + m];
        v[0] += d * d;
    }
    block_sum<1>(v, red);
    if (threadIdx.x == 0) loss[z] = (accumulate ? loss[z] : 0.0) + v[0] / B;
}

__global__ void to_bf16_kernel(const float *__restrict__ x, __nv_bfloat16 *__restrict__ y, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

// Epilogues of the tensor-core products (it_tc.cuh), called by a whole warp
// for its 32 x 16 block: lane holds row mw + lane, columns n0 .. n0+15.  Every
// global access goes through the warp's shared-memory scratch, so that
// consecutive lanes touch consecutive bytes of a row (a lane that walked its
// own row touched 32 rows per access).
using tc::NC;

// float rows of the block: lane l of access j holds columns 4 (l mod 4) .. of
// row 8 j + l / 4, both here and in the scratch (pitch 20: 16-byte aligned)
struct Rows { float4 r[4]; };

__device__ __forceinline__ Rows load_rows(const float *src, long long ld, int lane, int rows) {
    Rows x;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = 8 * j + (lane >> 2);
        x.r[j] = r < rows ? *reinterpret_cast<const float4 *>(src + r * ld + 4 * (lane & 3)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    return x;
}

// the lane's own row out of the scratch
__device__ __forceinline__ void lane_row(const float *scratch, int lane, float (&v)[NC]) {
#pragma unroll
    for (int q = 0; q < NC; q += 4) {
        const float4 t = *reinterpret_cast<const float4 *>(scratch + lane * 20 + q);
        v[q] = t.x; v[q + 1] = t.y; v[q + 2] = t.z; v[q + 3] = t.w;
    }
}

// the rows as loaded -> lane's own row
__device__ __forceinline__ void rows_to_lane(const Rows &x, int lane, float (&v)[NC], float *scratch) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
        *reinterpret_cast<float4 *>(scratch + (8 * j + (lane >> 2)) * 20 + 4 * (lane & 3)) = x.r[j];
    __syncwarp();
    lane_row(scratch, lane, v);
    __syncwarp();
}

// lane's own row -> rows of dst
__device__ __forceinline__ void store_rows(const float (&v)[NC], int lane, int rows, float *dst, long long ld,
                                           float *scratch) {
#pragma unroll
    for (int q = 0; q < NC; q += 4)
        *reinterpret_cast<float4 *>(scratch + lane * 20 + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = 8 * j + (lane >> 2);
        if (r < rows)
            *reinterpret_cast<float4 *>(dst + r * ld + 4 * (lane & 3)) =
                *reinterpret_cast<const float4 *>(scratch + r * 20 + 4 * (lane & 3));
    }
    __syncwarp();
}

// two bf16 in one register, the first in the low half
__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b) {
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// the same for bf16 (lane's row in a as pairs): 2 lanes per row
__device__ __forceinline__ void store_rows(const uint32_t (&a)[NC / 2], int lane, int rows, __nv_bfloat16 *dst,
                                           long long ld, float *scratch) {
    uint32_t *t = reinterpret_cast<uint32_t *>(scratch);   // pitch 12 words
#pragma unroll
    for (int q = 0; q < NC / 2; q += 4)
        *reinterpret_cast<uint4 *>(t + lane * 12 + q) = make_uint4(a[q], a[q + 1], a[q + 2], a[q + 3]);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = 16 * j + (lane >> 1);
        if (r < rows)
            *reinterpret_cast<uint4 *>(dst + r * ld + 8 * (lane & 1)) =
                *reinterpret_cast<const uint4 *>(t + r * 12 + 4 * (lane & 1));
    }
    __syncwarp();
}

// the block transposed: row c of dst (ld apart) gets column c
__device__ __forceinline__ void store_transposed(const uint32_t (&a)[NC / 2], int lane, int rows, __nv_bfloat16 *dst,
                                                 long long ld, float *scratch) {
    __nv_bfloat16 *t = reinterpret_cast<__nv_bfloat16 *>(scratch);   // [16 columns][40]
#pragma unroll
    for (int q = 0; q < NC / 2; ++q) {
        t[(2 * q) * 40 + lane] = __ushort_as_bfloat16((unsigned short)(a[q] & 0xffffu));
        t[(2 * q + 1) * 40 + lane] = __ushort_as_bfloat16((unsigned short)(a[q] >> 16));
    }
    __syncwarp();
    if (rows >= 32) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = 8 * j + (lane >> 2);
            *reinterpret_cast<uint4 *>(dst + r * ld + 8 * (lane & 3)) =
                *reinterpret_cast<const uint4 *>(t + r * 40 + 8 * (lane & 3));
        }
    } else {
        for (int c = lane >> 4; c < NC; c += 2)
            for (int r = lane & 15; r < rows; r += 16) dst[c * ld + r] = t[c * 40 + r];
    }
    __syncwarp();
}

// forward: Z = D + bias, Act = bf16(SiLU(Z)), and optionally Act transposed
struct TcFwd {
    const float *bias;
    long long zbias;
    float *Z;             // NULL: prediction, which needs neither Z nor ActT
    long long zact;
    __nv_bfloat16 *Act;   // [member][row][hi 0..H-1 | lo H..2H-1]
    long long zA;
    __nv_bfloat16 *ActT;
    long long zT, ldT;
    __device__ __forceinline__ float load(int z, int, int lane, int, int n0) const {
        return bias[z * zbias + n0 + (lane & (NC - 1))];
    }
    __device__ __forceinline__ void done(int z, int mw, int lane, int M, int n0, float (&v)[NC], float *scratch,
                                         float b) const {
        const int rows = M - mw;   // <= 0: a block past the batch
        if (rows <= 0) return;
        uint32_t hi[NC / 2], lo[NC / 2];
#pragma unroll
        for (int q = 0; q < NC; q += 2) {
            __nv_bfloat16 h[2], l[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                v[q + e] += __shfl_sync(0xffffffffu, b, q + e);
                const float s = silu(v[q + e]);
                h[e] = __float2bfloat16_rn(s);
                l[e] = __float2bfloat16_rn(s - __bfloat162float(h[e]));
            }
            hi[q / 2] = pack2(h[0], h[1]);
            lo[q / 2] = pack2(l[0], l[1]);
        }
        if (Z) store_rows(v, lane, rows, Z + z * zact + (long long)mw * H + n0, H, scratch);
        __nv_bfloat16 *act = Act + z * zA + (long long)mw * 2 * H + n0;
        store_rows(hi, lane, rows, act, 2 * H, scratch);
        store_rows(lo, lane, rows, act + H, 2 * H, scratch);
        if (ActT) store_transposed(hi, lane, rows, ActT + z * zT + (long long)n0 * ldT + mw, ldT, scratch);
    }
};

// data gradient: dZ = D * SiLU'(Z of the layer below), as fp32, bf16 and
// bf16 transposed
struct TcBwd {
    const float *Zp;
    float *dZ;
    __nv_bfloat16 *dZb;
    long long zact;
    __nv_bfloat16 *dZbT;
    long long zT, ldT;
    __device__ __forceinline__ Rows load(int z, int mw, int lane, int M, int n0) const {
        return load_rows(Zp + z * zact + (long long)mw * H + n0, H, lane, M - mw);
    }
    __device__ __forceinline__ void done(int z, int mw, int lane, int M, int n0, float (&v)[NC], float *scratch,
                                         const Rows &pre) const {
        const int rows = M - mw;
        if (rows <= 0) return;
        float zp[NC];
        rows_to_lane(pre, lane, zp, scratch);
        uint32_t db[NC / 2];
#pragma unroll
        for (int q = 0; q < NC; q += 2) {
            v[q] = v[q] * dsilu(zp[q]);
            v[q + 1] = v[q + 1] * dsilu(zp[q + 1]);
            db[q / 2] = pack2(__float2bfloat16_rn(v[q]), __float2bfloat16_rn(v[q + 1]));
        }
        const long long o = z * zact + (long long)mw * H + n0;
        store_rows(v, lane, rows, dZ + o, H, scratch);
        store_rows(db, lane, rows, dZb + o, H, scratch);
        store_transposed(db, lane, rows, dZbT + z * zT + (long long)n0 * ldT + mw, ldT, scratch);
    }
};

// weight gradient [out][in] into the member's gradient vector (P is odd, so a
// member's rows have no 16-byte alignment: 16 consecutive floats of two rows
// per store)
struct TcWgrad {
    float *grad;
    long long off;
    __device__ __forceinline__ int load(int, int, int, int, int) const { return 0; }
    __device__ __forceinline__ void done(int z, int mw, int lane, int M, int n0, float (&v)[NC], float *scratch,
                                         int) const {
#pragma unroll
        for (int q = 0; q < NC; ++q) scratch[lane * 17 + q] = v[q];
        __syncwarp();
        float *g = grad + z * P + off + (long long)mw * H + n0 + (lane & 15);
#pragma unroll 8
        for (int r = lane >> 4; r < 32; r += 2)
            if (mw + r < M) g[(long long)r * H] = scratch[r * 17 + (lane & 15)];
        __syncwarp();
    }
};

// Layer 1 forward: the 6 inputs as [hi 6 | lo 6] against [W1 | W1], one
// 16-wide k-step (4 columns of zeros) on mma.sync, fragments straight from
// global memory, and the forward epilogue of the other layers.  A warp owns
// 32 samples x 16 outputs.  In training the first thread moves the mini-batch
// counter on (the gather before this kernel has read it).
__global__ void __launch_bounds__(128)
layer1_fwd_kernel(const __nv_bfloat16 *__restrict__ A0, long long zA0, const __nv_bfloat16 *__restrict__ w1d, int B,
                  const TcFwd epi, int *__restrict__ batch) {
    __shared__ __align__(16) float scratch[4][tc::SCRATCH];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, z = blockIdx.z;
    if (batch && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 && z == 0) *batch += 1;
    const int mw = blockIdx.y * 32, n0 = (blockIdx.x * 4 + warp) * NC;
    const int grp = lane >> 2, tig = lane & 3;
    const __nv_bfloat16 *A = A0 + z * zA0, *W = w1d + (long long)z * H * 2 * NIN;
    const float bias = epi.load(z, mw, lane, B, n0);
    // pair k, k + 1 (k even) of a row of 12: zero past the row or the batch
    auto pair = [](const __nv_bfloat16 *row, int k, bool in) {
        return in && k < 2 * NIN ? *reinterpret_cast<const uint32_t *>(row + k) : 0u;
    };
    uint32_t af[2][4], bf[NC / 8][2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const int r = mw + a * 16 + grp;
        const __nv_bfloat16 *r0 = A + (long long)r * 2 * NIN, *r8 = r0 + 8 * 2 * NIN;
        af[a][0] = pair(r0, 2 * tig, r < B);
        af[a][1] = pair(r8, 2 * tig, r + 8 < B);
        af[a][2] = pair(r0, 2 * tig + 8, r < B);
        af[a][3] = pair(r8, 2 * tig + 8, r + 8 < B);
    }
#pragma unroll
    for (int b = 0; b < NC / 8; ++b) {
        const __nv_bfloat16 *c = W + (long long)(n0 + b * 8 + grp) * 2 * NIN;
        bf[b][0] = pair(c, 2 * tig, true);
        bf[b][1] = pair(c, 2 * tig + 8, true);
    }
    float *sc = scratch[warp];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < NC / 8; ++b) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            mma16816(c, af[a], bf[b]);
            float *o = sc + (a * 16 + grp) * 20 + b * 8 + 2 * tig;
            o[0] = c[0]; o[1] = c[1];
            o[8 * 20] = c[2]; o[8 * 20 + 1] = c[3];
        }
    __syncwarp();
    float v[NC];
    lane_row(sc, lane, v);
    __syncwarp();
    epi.done(z, mw, lane, B, n0, v, sc, bias);
}

// Layer 1 weight gradient gW1[o][i] = sum_m dZ1[m][o] A0[m][i] (bf16 hi part of
// the inputs): 256 x 6 outputs, so a block owns 16 rows o and the six columns
// of one 16 x 8 product.  Its four warps stage 256 samples at a time in shared
// memory (dZ1 from its transposed copy), one of them walks them 16 at a step
// (fragments straight from global memory by one warp took 11 us, this 4.2).
constexpr int W1_K = 256;
__global__ void __launch_bounds__(128)
layer1_wgrad_kernel(const __nv_bfloat16 *__restrict__ dZT, long long zT, long long ldT,
                    const __nv_bfloat16 *__restrict__ A0, long long zA0, int B, float *__restrict__ grad) {
    __shared__ __align__(16) __nv_bfloat16 ds[16][W1_K + 8];
    __shared__ __align__(16) unsigned short as[W1_K * 2 * NIN];
    const int tid = threadIdx.x, lane = tid & 31, z = blockIdx.y, o0 = blockIdx.x * 16;
    const int grp = lane >> 2, tig = lane & 3;
    const __nv_bfloat16 *D = dZT + z * zT + (long long)o0 * ldT;
    const uint32_t *A = reinterpret_cast<const uint32_t *>(A0 + z * zA0);   // 6 words per sample
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = 0; k0 < B; k0 += W1_K) {
        const int kn = min(W1_K, B - k0);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 16 * W1_K / 8 / 128; ++q) {
            const int e = tid + q * 128, r = e / (W1_K / 8), k = (e % (W1_K / 8)) * 8;
            if (k < kn)   // rows are padded to whole 64 samples
                *reinterpret_cast<uint4 *>(&ds[r][k]) = *reinterpret_cast<const uint4 *>(D + r * ldT + k0 + k);
        }
        for (int e = tid; e < kn * NIN; e += 128)
            reinterpret_cast<uint32_t *>(as)[e] = A[(long long)k0 * NIN + e];
        __syncthreads();
        if (tid < 32) {
            auto pair = [&](int r, int k) -> uint32_t {   // samples k, k + 1 (k even) of row r
                if (k >= kn) return 0u;
                const uint32_t v = *reinterpret_cast<const uint32_t *>(&ds[r][k]);
                return k + 1 < kn ? v : v & 0xffffu;
            };
            auto inputs = [&](int k) -> uint32_t {   // input grp of samples k, k + 1
                if (grp >= NIN) return 0u;
                const uint32_t lo = k < kn ? as[k * 2 * NIN + grp] : 0u;
                const uint32_t hi = k + 1 < kn ? as[(k + 1) * 2 * NIN + grp] : 0u;
                return lo | (hi << 16);
            };
#pragma unroll 4
            for (int kk = 0; kk < kn; kk += 16) {
                const int k = kk + 2 * tig;
                const uint32_t af[4] = {pair(grp, k), pair(grp + 8, k), pair(grp, k + 8), pair(grp + 8, k + 8)};
                const uint32_t bf[2] = {inputs(k), inputs(k + 8)};
                mma16816(c, af, bf);
            }
        }
    }
    if (tid < 32 && 2 * tig < NIN) {
        float *g = grad + z * P + OW1 + (long long)(o0 + grp) * NIN;
        g[2 * tig] = c[0];
        g[2 * tig + 1] = c[1];
        g[8 * NIN + 2 * tig] = c[2];
        g[8 * NIN + 2 * tig + 1] = c[3];
    }
}

// Adam (Kingma & Ba) on the FP32 master weights, refreshing the bf16 weights
// and their copies for the products: W2..W4 as [member][layer][out][W | W]
// along K (the forward's A operand is [hi | lo]) and transposed as
// [member][layer][in][out] (data gradient), by 32 x 32 tiles through shared
// memory so that every write is coalesced; W1 as [member][out][W1 | W1].
// Grid (H/32, 3 H/32 + 1, members), block (32, 8): the extra row of blocks
// takes W1, the biases and the output layer.  UPDATE = false only packs.
// step: the bias corrections of this step are corr[*step] (the counter lives
// on the device, so that a recorded step can be replayed).
struct AdamArgs {
    float *master;
    const float *g;
    float *m1, *m2;
    float lr, b1, b2, eps;
    const float2 *corr;
    const int *step;
};

template <bool UPDATE>
__device__ __forceinline__ __nv_bfloat16 adam_one(const AdamArgs &a, __nv_bfloat16 *w, long long i, float c1, float c2) {
    if (!UPDATE) return w[i];
    const float gi = a.g[i];
    const float m1 = a.b1 * a.m1[i] + (1.f - a.b1) * gi;
    const float m2 = a.b2 * a.m2[i] + (1.f - a.b2) * gi * gi;
    a.m1[i] = m1;
    a.m2[i] = m2;
    const float p = a.master[i] - a.lr * (m1 / c1) / (sqrtf(m2 / c2) + a.eps);
    a.master[i] = p;
    const __nv_bfloat16 v = __float2bfloat16_rn(p);
    w[i] = v;
    return v;
}

template <bool UPDATE>
__global__ void __launch_bounds__(256)
adam_pack_kernel(const AdamArgs a, __nv_bfloat16 *__restrict__ w, __nv_bfloat16 *__restrict__ wt,
                 __nv_bfloat16 *__restrict__ wtt, __nv_bfloat16 *__restrict__ w1d) {
    __shared__ __nv_bfloat16 tile[32][34];
    const long long z = blockIdx.z;
    float c1 = 1.f, c2 = 1.f;
    if (UPDATE) {
        const float2 c = a.corr[*a.step];
        c1 = c.x;
        c2 = c.y;
    }
    if (blockIdx.y == 3 * (H / 32)) {
        const int tid = threadIdx.y * 32 + threadIdx.x;
        for (int e = blockIdx.x * 256 + tid; e < H * NIN; e += (H / 32) * 256) {
            const int o = e / NIN, i = e - o * NIN;
            const __nv_bfloat16 v = adam_one<UPDATE>(a, w, z * P + OW1 + e, c1, c2);
            w1d[(z * H + o) * 2 * NIN + i] = v;
            w1d[(z * H + o) * 2 * NIN + NIN + i] = v;
        }
        if (UPDATE) {
            // biases of the four hidden layers, output weights and bias
            const int e = blockIdx.x * 256 + tid;
            const long long at = e < H          ? OB1 + e
                                 : e < 2 * H    ? OB2 + (e - H)
                                 : e < 3 * H    ? OB3 + (e - 2 * H)
                                 : e < 4 * H    ? OB4 + (e - 3 * H)
                                 : e <= 5 * H   ? OW5 + (e - 4 * H)
                                                : -1;
            if (at >= 0) (void)adam_one<UPDATE>(a, w, z * P + at, c1, c2);
        }
        return;
    }
    const int l = blockIdx.y / (H / 32), to = blockIdx.y % (H / 32), ti = blockIdx.x;
    const long long src = z * P + OW2 + (long long)l * (H * H + H);
    const long long blk = (z * 3 + l) * H * H;
#pragma unroll
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int o = to * 32 + j, i = ti * 32 + threadIdx.x;
        const __nv_bfloat16 v = adam_one<UPDATE>(a, w, src + o * H + i, c1, c2);
        tile[j][threadIdx.x] = v;
        wt[2 * blk + (long long)o * 2 * H + i] = v;
        wt[2 * blk + (long long)o * 2 * H + H + i] = v;
    }
    __syncthreads();
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int i = ti * 32 + j, o = to * 32 + threadIdx.x;
        wtt[blk + i * H + o] = tile[threadIdx.x][j];
    }
}

// normalised bf16 inputs of a batch for every member:
// A0[z][m][j] = hi and A0[z][m][6 + j] = lo of (x[idx[z][m]][j] - mean[j]) / std[j], yb[z][m] = y[idx[z][m]]
// (idx == NULL: sample m for every member)
__global__ void gather_inputs_kernel(const float *__restrict__ X, const float *__restrict__ Y,
                                     const int *__restrict__ idx, long long istride, int *__restrict__ count,
                                     int B, int members, int bmax, const float *__restrict__ mean, const float *__restrict__ inv_std,
                                     __nv_bfloat16 *__restrict__ A0, float *__restrict__ yb) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx && e == 0) count[0] += 1;   // the step (its Adam update reads it); count[1] is the mini-batch
    if (e >= (long long)members * B * NIN) return;
    const int z = (int)(e / ((long long)B * NIN));
    const int r0 = (int)(e - (long long)z * B * NIN);
    const int m = r0 / NIN, j = r0 % NIN;
    const int r = idx ? idx[z * istride + (long long)count[1] * B + m] : m;
    const float x = (X[(long long)r * NIN + j] - mean[j]) * inv_std[j];
    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
    A0[((long long)z * bmax + m) * 2 * NIN + j] = hi;
    A0[((long long)z * bmax + m) * 2 * NIN + NIN + j] = __float2bfloat16_rn(x - __bfloat162float(hi));
    if (j == 0 && Y) yb[z * bmax + m] = Y[r];
}

}  // namespace mlp
}  // namespace itk

using namespace itk;
using namespace itk::mlp;

struct it_mlp {
    int members, bmax;
    float *master, *grad, *m1, *m2;
    __nv_bfloat16 *w;
    long long adam_t;
    float *mean, *inv_std;        // device [6]
    double h_mean[NIN], h_std[NIN];
    // batch workspace (per member strides zact = bmax * H)
    __nv_bfloat16 *A0;            // [member][bmax][hi 6 | lo 6]
    float *Z[4];
    __nv_bfloat16 *Act[4];        // [member][bmax][hi 256 | lo 256]
    float *dZ[2];
    __nv_bfloat16 *dZb[2];
    float *fhat, *dz, *yb;
    double *loss;
    // tensor-core operands: W2..W4 as [member][layer][out][in] and
    // [member][layer][in][out], A1..A3 transposed and the bf16 error signal
    // transposed, [member][256][bpad] (bpad: max_batch rounded up to 64)
    __nv_bfloat16 *wt, *wtt, *actT[3], *dzbT[2];
    __nv_bfloat16 *w1d;           // [member][256][W1 | W1] for the layer-1 product with [hi | lo] inputs
    long long bpad;
    int *d_err;                   // a bounded wait of the tensor-core kernel ran out
    int *eidx;                    // [members][n_data]: every member's sample order of one epoch
    long long eidx_cap;
    double *eloss;                // [members]: the epoch's summed batch losses
    int *count;                   // {step of the call, mini-batch of the epoch}
    float2 *corr;                 // Adam's bias corrections of a call's steps
    long long corr_cap;
    float *pX;                    // inputs of a call, kept between calls up to kKeepInputs
    long long pX_cap;
    cudaStream_t side[2];         // weight and bias gradients run beside the data gradients
    cudaEvent_t ev[12];
    int refuse_recording;         // test hook: a recorded step is never instantiated
    cudaEvent_t up[2];            // the uploads of an epoch have been read (epochs alternate)
    // training set
    float *X, *Y;
    long long n_data;
    cudaStream_t stream;
};

namespace {

int mfail(int code, const std::string &m) {
    set_error(m);
    return code;
}

void mlp_free(it_mlp *n) {
    if (!n) return;
    if (n->stream) cudaStreamSynchronize(n->stream);
    cudaFree(n->master); cudaFree(n->grad); cudaFree(n->m1); cudaFree(n->m2); cudaFree(n->w);
    cudaFree(n->mean); cudaFree(n->inv_std); cudaFree(n->A0);
    for (int l = 0; l < 4; ++l) { cudaFree(n->Z[l]); cudaFree(n->Act[l]); }
    for (int q = 0; q < 2; ++q) { cudaFree(n->dZ[q]); cudaFree(n->dZb[q]); }
    cudaFree(n->fhat); cudaFree(n->dz); cudaFree(n->yb); cudaFree(n->loss);
    cudaFree(n->eidx); cudaFree(n->eloss); cudaFree(n->count); cudaFree(n->corr); cudaFree(n->pX);
    for (auto &e : n->ev)
        if (e) cudaEventDestroy(e);
    for (auto &e : n->up)
        if (e) cudaEventDestroy(e);
    for (auto &v : n->side)
        if (v) cudaStreamDestroy(v);
    cudaFree(n->wt); cudaFree(n->wtt); cudaFree(n->w1d); cudaFree(n->d_err);
    for (int q = 0; q < 3; ++q) cudaFree(n->actT[q]);
    for (int q = 0; q < 2; ++q) cudaFree(n->dzbT[q]);
    cudaFree(n->X); cudaFree(n->Y);
    if (n->stream) cudaStreamDestroy(n->stream);
    delete n;
}

const long long kOffW[4] = {OW1, OW2, OW3, OW4};
const long long kOffB[4] = {OB1, OB2, OB3, OB4};

// D = A B^T on the tensor cores for every member: A [members][M rows][K],
// B [members][N rows][K] (bf16, K contiguous, byte strides of a row and of a
// member), N a multiple of 32
template <class Epi>
int launch_tc(it_mlp *n, const void *A, long long a_row, long long a_mem, const void *Bm, long long b_row,
              long long b_mem, int M, int N, int K, const Epi &epi, cudaStream_t s) {
    CUtensorMap ta, tb;
    int rc = encode_bf16_sw128(&ta, A, K, M, n->members, a_row, a_mem, tc::TM);
    if (!rc) rc = encode_bf16_sw128(&tb, Bm, K, N, n->members, b_row, b_mem, tc::TN);
    if (rc) return rc;
    dim3 grid(N / tc::TN, (M + tc::TM - 1) / tc::TM, n->members);
    tc::tc_gemm_kernel<Epi><<<grid, tc::THREADS, tc::SMEM_BYTES, s>>>(ta, tb, M, N, K, epi, n->d_err);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// forward of B samples already in A0 (and yb when training)
int forward(it_mlp *n, int B, bool train) {
    const long long zact = (long long)n->bmax * H, zA = 2 * zact, zT = (long long)H * n->bpad;
    // layer 1 (6 inputs as hi | lo against W1 | W1)
    {
        TcFwd e{n->master + kOffB[0], P, train ? n->Z[0] : nullptr, zact, n->Act[0], zA, train ? n->actT[0] : nullptr,
                zT, n->bpad};
        layer1_fwd_kernel<<<dim3(H / (4 * NC), (B + 31) / 32, n->members), 128, 0, n->stream>>>(
            n->A0, (long long)n->bmax * 2 * NIN, n->w1d, B, e, train ? n->count + 1 : nullptr);
        IT_CK(cudaGetLastError());
    }
    // layers 2-4 on the tensor cores: [hi | lo] (K = 512) against [W | W]
    for (int l = 1; l < 4; ++l) {
        TcFwd e{n->master + kOffB[l], P, train ? n->Z[l] : nullptr, zact, n->Act[l], zA,
                train && l < 3 ? n->actT[l] : nullptr, zT, n->bpad};
        int rc = launch_tc(n, n->Act[l - 1], 4LL * H, 2LL * zA, n->wt + (long long)(l - 1) * H * 2 * H, 4LL * H,
                           2LL * 3 * H * 2 * H, B, H, 2 * H, e, n->stream);
        if (rc) return rc;
    }
    dim3 grid((B + 7) / 8, n->members);
    out_layer_kernel<<<grid, 256, 0, n->stream>>>(n->Act[3], n->Z[3], n->w, n->master, n->yb, n->bmax, B, train ? 1 : 0,
                                                  n->fhat, n->dz, n->dZ[0], n->dZb[0], zact, n->dzbT[0], zT, n->bpad,
                                                  zA);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// backward of the batch into n->grad (after forward(train = true)).  The data
// gradients form the chain; what only reads a layer's error signal runs beside
// it, the weight gradients on one side stream, the bias and output-layer
// gradients and the loss on another, ordered by events: a layer's error
// signal buffer is written again two layers further down, after both side
// streams have read it.
int backward(it_mlp *n, int B, double *loss, bool accumulate) {
    const long long zact = (long long)n->bmax * H, zA = 2 * zact, zT = (long long)H * n->bpad;
    cudaStream_t sw = n->side[0], sb = n->side[1];
    // events: ready[l] the error signal of layer l is complete, wread[l] /
    // bread[l] the weight / bias gradient of layer l has been formed
    cudaEvent_t *ready = n->ev, *wread = n->ev + 4, *bread = n->ev + 8;
    auto bias = [&](int l, int buf) -> int {
        bias_grad_kernel<<<dim3(H / 32, n->members), 256, 0, sb>>>(n->dZ[buf], B, n->grad, kOffB[l], zact);
        IT_CK(cudaGetLastError());
        return IT_OK;
    };
    int cur = 0, rc = IT_OK;
    for (int l = 3; l >= 1; --l) {
        IT_CK(cudaEventRecord(ready[l], n->stream));
        IT_CK(cudaStreamWaitEvent(sw, ready[l], 0));
        IT_CK(cudaStreamWaitEvent(sb, ready[l], 0));
        // data gradient into the layer below: dZ_{l-1} = (dZ_l W_l) * SiLU'(Z_{l-1})
        if (l < 3) {   // the buffer it writes has been read
            IT_CK(cudaStreamWaitEvent(n->stream, wread[l + 1], 0));
            IT_CK(cudaStreamWaitEvent(n->stream, bread[l + 1], 0));
        }
        TcBwd d{n->Z[l - 1], n->dZ[cur ^ 1], n->dZb[cur ^ 1], zact, n->dzbT[cur ^ 1], zT, n->bpad};
        rc = launch_tc(n, n->dZb[cur], 2LL * H, 2LL * zact, n->wtt + (long long)(l - 1) * H * H, 2LL * H,
                       2LL * 3 * H * H, B, H, H, d, n->stream);
        if (rc) return rc;
        // weight gradient gW[o][i] = sum_m dZ[m][o] A_{l-1}[m][i] (bf16 hi part of
        // the activation): the K = batch axis is contiguous in the transposed copies
        TcWgrad w{n->grad, kOffW[l]};
        rc = launch_tc(n, n->dzbT[cur], 2LL * n->bpad, 2LL * zT, n->actT[l - 1], 2LL * n->bpad, 2LL * zT, H, H, B, w,
                       sw);
        if (!rc) rc = bias(l, cur);
        if (rc) return rc;
        IT_CK(cudaEventRecord(wread[l], sw));
        IT_CK(cudaEventRecord(bread[l], sb));
        cur ^= 1;
    }
    // the error signal of layer 1, and what the output layer left
    IT_CK(cudaEventRecord(ready[0], n->stream));
    IT_CK(cudaStreamWaitEvent(sb, ready[0], 0));
    layer1_wgrad_kernel<<<dim3(H / 16, n->members), 128, 0, n->stream>>>(
        n->dzbT[cur], zT, n->bpad, n->A0, (long long)n->bmax * 2 * NIN, B, n->grad);
    IT_CK(cudaGetLastError());
    rc = bias(0, cur);
    if (rc) return rc;
    out_grad_kernel<<<dim3(H / 32, n->members), 256, 0, sw>>>(n->Act[3], n->dz, B, n->grad, zA);
    IT_CK(cudaGetLastError());
    if (loss) {
        loss_kernel<<<n->members, 256, 0, sb>>>(n->fhat, n->yb, n->bmax, B, loss, accumulate);
        IT_CK(cudaGetLastError());
    }
    IT_CK(cudaEventRecord(wread[0], sw));
    IT_CK(cudaEventRecord(bread[0], sb));
    IT_CK(cudaStreamWaitEvent(n->stream, wread[0], 0));
    IT_CK(cudaStreamWaitEvent(n->stream, bread[0], 0));
    return IT_OK;
}

// the bf16 tensor-core copies of W2..W4 after the bf16 weights changed
int pack_weights(it_mlp *n) {
    adam_pack_kernel<false><<<dim3(H / 32, 3 * (H / 32) + 1, n->members), dim3(32, 8), 0, n->stream>>>(
        AdamArgs{}, n->w, n->wt, n->wtt, n->w1d);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// IT_ETIMEOUT if a bounded wait of the tensor-core kernel ran out (the flag
// is cleared)
int check_device_error(it_mlp *n) {
    int err = 0;
    IT_CK(cudaMemcpyAsync(&err, n->d_err, sizeof(int), cudaMemcpyDeviceToHost, n->stream));
    IT_CK(cudaStreamSynchronize(n->stream));
    if (err) {
        IT_CK(cudaMemsetAsync(n->d_err, 0, sizeof(int), n->stream));
        return mfail(IT_ETIMEOUT, "a bounded wait of the tensor-core GEMM ran out");
    }
    return IT_OK;
}

// Floats of a call's inputs that a network keeps room for; larger calls
// allocate and free theirs.
constexpr long long kKeepInputs = 1 << 20;

// The inputs (and targets) of a call on the device: in the network's buffer
// when they fit it (*own = false), else in memory the caller frees.
int upload_inputs(it_mlp *n, long long count, const double *x, const double *y, float **dX, float **dY, bool *own) {
    const long long nx = count * NIN, ny = y ? count : 0;
    std::vector<float> h((size_t)(nx + ny));
    for (long long i = 0; i < nx; ++i) h[i] = (float)x[i];
    for (long long i = 0; i < ny; ++i) h[nx + i] = (float)y[i];
    *own = nx + ny > kKeepInputs;
    float *d = nullptr;
    if (*own) {
        IT_CK(cudaMalloc(&d, sizeof(float) * (nx + ny)));
    } else {
        if (nx + ny > n->pX_cap) {
            cudaFree(n->pX);
            n->pX = nullptr;
            n->pX_cap = 0;
            IT_CK(cudaMalloc(&n->pX, sizeof(float) * (nx + ny)));
            n->pX_cap = nx + ny;
        }
        d = n->pX;
    }
    *dX = d;
    if (dY) *dY = y ? d + nx : nullptr;
    cudaError_t e = cudaMemcpyAsync(d, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);   // h is released on return
    if (e != cudaSuccess) {
        if (*own) cudaFree(d);
        return cuda_fail(e, "network inputs");
    }
    return IT_OK;
}

// idx: per member the sample rows in the order of an epoch, member z's at
// idx + z istride, the mini-batch of B rows count[1] of it (NULL: rows 0..B-1)
int gather(it_mlp *n, const float *X, const float *Y, const int *idx, long long istride, int B) {
    const long long tot = (long long)n->members * B * NIN;
    gather_inputs_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, n->stream>>>(
        X, Y, idx, istride, n->count, B, n->members, n->bmax, n->mean, n->inv_std, n->A0, n->yb);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// Room for the bias corrections of `steps` Adam steps.
int adam_room(it_mlp *n, long long steps) {
    if (steps <= n->corr_cap) return IT_OK;
    cudaFree(n->corr);
    n->corr = nullptr;
    n->corr_cap = 0;
    IT_CK(cudaMalloc(&n->corr, sizeof(float2) * steps));
    n->corr_cap = steps;
    return IT_OK;
}

// The bias corrections of the next `steps` Adam steps; the counters restart:
// the step at `first` (-1 where a gather raises it before its first use), the
// mini-batch at 0.  The copy out of c is asynchronous (pageable memory is only
// staged where it has to be, and a Grace host's pages need not): the caller
// keeps c unchanged until the stream has passed it.
int adam_begin(it_mlp *n, long long steps, int first, std::vector<float2> &c) {
    int rc = adam_room(n, steps);
    if (rc) return rc;
    c.resize((size_t)steps);
    for (long long q = 0; q < steps; ++q) {
        const double t = (double)(n->adam_t + 1 + q);
        c[q] = make_float2((float)(1.0 - std::pow(0.9, t)), (float)(1.0 - std::pow(0.999, t)));
    }
    IT_CK(cudaMemcpyAsync(n->corr, c.data(), sizeof(float2) * steps, cudaMemcpyHostToDevice, n->stream));
    IT_CK(cudaMemsetAsync(n->count, first < 0 ? 0xff : 0, sizeof(int), n->stream));
    IT_CK(cudaMemsetAsync(n->count + 1, 0, sizeof(int), n->stream));
    return IT_OK;
}

int adam_step(it_mlp *n, float lr) {
    AdamArgs a{n->master, n->grad, n->m1, n->m2, lr, 0.9f, 0.999f, 1e-8f, n->corr, n->count};
    adam_pack_kernel<true><<<dim3(H / 32, 3 * (H / 32) + 1, n->members), dim3(32, 8), 0, n->stream>>>(
        a, n->w, n->wt, n->wtt, n->w1d);
    IT_CK(cudaGetLastError());
    return IT_OK;
}

// one training step on mini-batch count[1] of the epoch order
int train_step(it_mlp *n, int B, float lr, double *loss, bool accumulate) {
    int rc = gather(n, n->X, n->Y, n->eidx, n->n_data, B);
    if (!rc) rc = forward(n, B, true);
    if (!rc) rc = backward(n, B, loss, accumulate);
    if (!rc) rc = adam_step(n, lr);
    return rc;
}

// A training step recorded as a graph: its launches have the same arguments
// every time (the step and mini-batch are counted on the device).
int record_step(it_mlp *n, int B, float lr, double *loss, cudaGraphExec_t *out) {
    cudaGraph_t g = nullptr;
    IT_CK(cudaStreamBeginCapture(n->stream, cudaStreamCaptureModeThreadLocal));
    const int rc = train_step(n, B, lr, loss, true);
    cudaError_t e = cudaStreamEndCapture(n->stream, &g);
    if (rc) { if (g) cudaGraphDestroy(g); return rc; }
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture(training step)");
    e = n->refuse_recording ? cudaErrorMemoryAllocation : cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) { *out = nullptr; return cuda_fail(e, "cudaGraphInstantiate(training step)"); }
    return IT_OK;
}

uint64_t splitmix_next(uint64_t &x) {
    uint64_t z = (x += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int it_mlp_create(int32_t members, int32_t max_batch, it_mlp **out) {
    if (!out) return mfail(IT_EINVAL, "out is NULL");
    *out = nullptr;
    if (members < 1 || members > 64 || max_batch < 1 || max_batch > (1 << 20))
        return mfail(IT_EINVAL, "members must be 1..64 and max_batch 1..2^20");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return mfail(IT_ECUDA, "no CUDA device available");
    it_mlp *n = new (std::nothrow) it_mlp();
    if (!n) return mfail(IT_ENOMEM, "host allocation failed");
    n->members = members;
    n->bmax = max_batch;
    const long long np = (long long)members * P, za = (long long)members * max_batch * H;
    cudaError_t e;
    auto bail = [&](const char *w) { int rc = cuda_fail(e, w); mlp_free(n); return rc; };
    if ((e = cudaStreamCreateWithFlags(&n->stream, cudaStreamNonBlocking)) != cudaSuccess) return bail("stream");
    if ((e = cudaMalloc(&n->master, sizeof(float) * np)) != cudaSuccess ||
        (e = cudaMalloc(&n->grad, sizeof(float) * np)) != cudaSuccess ||
        (e = cudaMalloc(&n->m1, sizeof(float) * np)) != cudaSuccess ||
        (e = cudaMalloc(&n->m2, sizeof(float) * np)) != cudaSuccess ||
        (e = cudaMalloc(&n->w, sizeof(__nv_bfloat16) * np)) != cudaSuccess ||
        (e = cudaMalloc(&n->mean, sizeof(float) * NIN)) != cudaSuccess ||
        (e = cudaMalloc(&n->inv_std, sizeof(float) * NIN)) != cudaSuccess ||
        (e = cudaMalloc(&n->A0, sizeof(__nv_bfloat16) * members * max_batch * 2 * NIN)) != cudaSuccess ||
        (e = cudaMalloc(&n->fhat, sizeof(float) * members * max_batch)) != cudaSuccess ||
        (e = cudaMalloc(&n->dz, sizeof(float) * members * max_batch)) != cudaSuccess ||
        (e = cudaMalloc(&n->yb, sizeof(float) * members * max_batch)) != cudaSuccess ||
        (e = cudaMalloc(&n->loss, sizeof(double) * members)) != cudaSuccess)
        return bail("mlp allocation");
    for (auto &v : n->side)
        if ((e = cudaStreamCreateWithFlags(&v, cudaStreamNonBlocking)) != cudaSuccess) return bail("mlp streams");
    if ((e = cudaMalloc(&n->count, 2 * sizeof(int))) != cudaSuccess ||
        (e = cudaMemsetAsync(n->count, 0, 2 * sizeof(int), n->stream)) != cudaSuccess)
        return bail("mlp step counters");
    for (auto &v : n->ev)
        if ((e = cudaEventCreateWithFlags(&v, cudaEventDisableTiming)) != cudaSuccess) return bail("mlp events");
    for (auto &v : n->up)
        if ((e = cudaEventCreateWithFlags(&v, cudaEventDisableTiming)) != cudaSuccess) return bail("mlp events");
    n->bpad = ((long long)max_batch + 63) / 64 * 64;
    const long long zw = (long long)members * 3 * H * H, zt = (long long)members * H * n->bpad;
    if ((e = cudaMalloc(&n->wt, sizeof(__nv_bfloat16) * 2 * zw)) != cudaSuccess ||
        (e = cudaMalloc(&n->w1d, sizeof(__nv_bfloat16) * members * H * 2 * NIN)) != cudaSuccess ||
        (e = cudaMalloc(&n->wtt, sizeof(__nv_bfloat16) * zw)) != cudaSuccess ||
        (e = cudaMalloc(&n->d_err, sizeof(int))) != cudaSuccess ||
        (e = cudaMemsetAsync(n->d_err, 0, sizeof(int), n->stream)) != cudaSuccess)
        return bail("mlp tensor-core operands");
    for (int q = 0; q < 3; ++q)
        if ((e = cudaMalloc(&n->actT[q], sizeof(__nv_bfloat16) * zt)) != cudaSuccess) return bail("mlp activations");
    for (int q = 0; q < 2; ++q)
        if ((e = cudaMalloc(&n->dzbT[q], sizeof(__nv_bfloat16) * zt)) != cudaSuccess) return bail("mlp gradients");
    if ((e = cudaFuncSetAttribute(tc::tc_gemm_kernel<TcFwd>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  tc::SMEM_BYTES)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(tc::tc_gemm_kernel<TcBwd>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  tc::SMEM_BYTES)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(tc::tc_gemm_kernel<TcWgrad>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  tc::SMEM_BYTES)) != cudaSuccess)
        return bail("cudaFuncSetAttribute(tensor-core GEMM)");
    for (int l = 0; l < 4; ++l)
        if ((e = cudaMalloc(&n->Z[l], sizeof(float) * za)) != cudaSuccess ||
            (e = cudaMalloc(&n->Act[l], sizeof(__nv_bfloat16) * 2 * za)) != cudaSuccess)
            return bail("mlp activations");
    for (int q = 0; q < 2; ++q)
        if ((e = cudaMalloc(&n->dZ[q], sizeof(float) * za)) != cudaSuccess ||
            (e = cudaMalloc(&n->dZb[q], sizeof(__nv_bfloat16) * za)) != cudaSuccess)
            return bail("mlp gradients");
    if ((e = cudaMemsetAsync(n->master, 0, sizeof(float) * np, n->stream)) != cudaSuccess ||
        (e = cudaMemsetAsync(n->w, 0, sizeof(__nv_bfloat16) * np, n->stream)) != cudaSuccess ||
        (e = cudaMemsetAsync(n->m1, 0, sizeof(float) * np, n->stream)) != cudaSuccess ||
        (e = cudaMemsetAsync(n->m2, 0, sizeof(float) * np, n->stream)) != cudaSuccess)
        return bail("mlp init");
    double mean[NIN] = {0}, sd[NIN] = {1, 1, 1, 1, 1, 1};
    *out = n;
    return it_mlp_set_normalization(n, mean, sd);
}

int it_mlp_set_params(it_mlp *n, int32_t member, const float *params, int64_t count) {
    if (!n || !params || member < 0 || member >= n->members || count != P) return mfail(IT_EINVAL, "bad argument");
    IT_CK(cudaMemcpyAsync(n->master + (long long)member * P, params, sizeof(float) * P, cudaMemcpyHostToDevice, n->stream));
    to_bf16_kernel<<<256, 256, 0, n->stream>>>(n->master + (long long)member * P, n->w + (long long)member * P, P);
    IT_CK(cudaGetLastError());
    if (int rc = pack_weights(n)) return rc;
    // a new starting point: the optimiser state restarts
    IT_CK(cudaMemsetAsync(n->m1 + (long long)member * P, 0, sizeof(float) * P, n->stream));
    IT_CK(cudaMemsetAsync(n->m2 + (long long)member * P, 0, sizeof(float) * P, n->stream));
    n->adam_t = 0;
    IT_CK(cudaStreamSynchronize(n->stream));
    return IT_OK;
}

int it_mlp_get_params(it_mlp *n, int32_t member, float *out, int64_t count) {
    if (!n || !out || member < 0 || member >= n->members || count != P) return mfail(IT_EINVAL, "bad argument");
    IT_CK(cudaMemcpyAsync(out, n->master + (long long)member * P, sizeof(float) * P, cudaMemcpyDeviceToHost, n->stream));
    IT_CK(cudaStreamSynchronize(n->stream));
    return IT_OK;
}

int it_mlp_set_normalization(it_mlp *n, const double *mean6, const double *std6) {
    if (!n || !mean6 || !std6) return mfail(IT_EINVAL, "bad argument");
    float m[NIN], is[NIN];
    for (int j = 0; j < NIN; ++j) {
        if (!(std::isfinite(mean6[j]) && std::isfinite(std6[j]) && std6[j] > 0)) return mfail(IT_EINVAL, "std must be > 0");
        n->h_mean[j] = mean6[j];
        n->h_std[j] = std6[j];
        m[j] = (float)mean6[j];
        is[j] = (float)(1.0 / std6[j]);
    }
    IT_CK(cudaMemcpyAsync(n->mean, m, sizeof(m), cudaMemcpyHostToDevice, n->stream));
    IT_CK(cudaMemcpyAsync(n->inv_std, is, sizeof(is), cudaMemcpyHostToDevice, n->stream));
    IT_CK(cudaStreamSynchronize(n->stream));
    return IT_OK;
}

int it_mlp_fit_normalization(it_mlp *n, int64_t count, const double *x) {
    if (!n || !x || count < 2) return mfail(IT_EINVAL, "need at least 2 samples");
    double mean[NIN] = {0}, sd[NIN] = {0};
    for (int64_t i = 0; i < count; ++i)
        for (int j = 0; j < NIN; ++j) mean[j] += x[i * NIN + j];
    for (int j = 0; j < NIN; ++j) mean[j] /= (double)count;
    for (int64_t i = 0; i < count; ++i)
        for (int j = 0; j < NIN; ++j) sd[j] += (x[i * NIN + j] - mean[j]) * (x[i * NIN + j] - mean[j]);
    for (int j = 0; j < NIN; ++j) {
        sd[j] = std::sqrt(sd[j] / (double)(count - 1));
        if (!(sd[j] > 0)) sd[j] = 1.0;
    }
    return it_mlp_set_normalization(n, mean, sd);
}

int it_mlp_set_data(it_mlp *n, int64_t count, const double *x, const double *y) {
    if (!n || !x || !y || count < 1 || count > 0x7fffffff) return mfail(IT_EINVAL, "bad argument");
    cudaFree(n->X); cudaFree(n->Y);
    n->X = n->Y = nullptr;
    n->n_data = 0;
    std::vector<float> hx((size_t)count * NIN), hy((size_t)count);
    for (long long i = 0; i < count * NIN; ++i) hx[i] = (float)x[i];
    for (long long i = 0; i < count; ++i) hy[i] = (float)y[i];
    IT_CK(cudaMalloc(&n->X, sizeof(float) * hx.size()));
    IT_CK(cudaMalloc(&n->Y, sizeof(float) * hy.size()));
    cudaError_t e = cudaMemcpyAsync(n->X, hx.data(), sizeof(float) * hx.size(), cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(n->Y, hy.data(), sizeof(float) * hy.size(), cudaMemcpyHostToDevice, n->stream);
    const cudaError_t done = cudaStreamSynchronize(n->stream);   // hx and hy are released on return, failed or not
    if (e == cudaSuccess) e = done;
    if (e != cudaSuccess) return cuda_fail(e, "training data");
    n->n_data = count;
    return IT_OK;
}

int it_mlp_train(it_mlp *n, int32_t epochs, int32_t batch, double lr, uint64_t seed, double *loss_per_epoch) {
    if (!n || epochs < 0 || batch < 1 || batch > n->bmax || !(lr > 0)) return mfail(IT_EINVAL, "bad argument");
    if (n->n_data < 1) return mfail(IT_ESTATE, "no training data (it_mlp_set_data)");
    const long long N = n->n_data;
    const int Z = n->members;
    if (n->eidx_cap < (long long)Z * N) {
        cudaFree(n->eidx);
        n->eidx = nullptr;
        n->eidx_cap = 0;
        IT_CK(cudaMalloc(&n->eidx, sizeof(int) * (size_t)Z * N));
        n->eidx_cap = (long long)Z * N;
    }
    if (!n->eloss) IT_CK(cudaMalloc(&n->eloss, sizeof(double) * Z));
    // each member walks the data in its own order (ensemble diversity); one
    // epoch's orders go to the device at once, and the batches of the epoch
    // are enqueued without host synchronisation
    std::vector<uint64_t> st(Z);
    for (int z = 0; z < Z; ++z) st[z] = seed + 0x9E3779B97F4A7C15ULL * (uint64_t)(z + 1);
    std::vector<double> lossb(Z);
    // mini-batches of an epoch: whole ones (the tail is left out), or one
    // short one when there are fewer samples than a batch
    const int B = (int)std::min<long long>(batch, N);
    const long long nb = std::max(1LL, N / batch);
    double *eloss = loss_per_epoch ? n->eloss : nullptr;
    int rc = adam_room(n, nb);
    if (rc) return rc;
    // host copies of what an epoch uploads (sample orders, Adam's corrections),
    // two of each: an epoch's are written again two epochs later, once its
    // uploads have been read
    std::vector<int> hidx[2];
    std::vector<float2> hcorr[2];
    for (int u = 0; u < std::min(epochs, 2); ++u) {
        hidx[u].resize((size_t)Z * N);
        hcorr[u].resize((size_t)nb);
    }
    // the same step over and over: recorded once and replayed where the
    // recording (about 0.4 ms) pays; a step that cannot be recorded (no memory
    // for the graph) is launched each time
    cudaGraphExec_t graph = nullptr;
    if (nb * epochs >= 8 && record_step(n, B, (float)lr, eloss, &graph)) {
        graph = nullptr;
        (void)cudaGetLastError();
    }
    cudaError_t e = cudaSuccess;
    for (int ep = 0; ep < epochs && !rc && e == cudaSuccess; ++ep) {
        const int u = ep & 1;
        if (ep >= 2) {
            e = cudaEventSynchronize(n->up[u]);
            if (e != cudaSuccess) break;
        }
        for (int z = 0; z < Z; ++z) {
            int *pz = hidx[u].data() + (size_t)z * N;
            for (long long i = 0; i < N; ++i) pz[i] = (int)i;
            for (long long i = N - 1; i > 0; --i) {   // Fisher-Yates with SplitMix64
                const long long j = (long long)(splitmix_next(st[z]) % (uint64_t)(i + 1));
                std::swap(pz[i], pz[j]);
            }
        }
        e = cudaMemcpyAsync(n->eidx, hidx[u].data(), sizeof(int) * (size_t)Z * N, cudaMemcpyHostToDevice, n->stream);
        if (e == cudaSuccess) rc = adam_begin(n, nb, -1, hcorr[u]);
        if (e == cudaSuccess && !rc) e = cudaEventRecord(n->up[u], n->stream);
        if (e == cudaSuccess && !rc && eloss) e = cudaMemsetAsync(eloss, 0, sizeof(double) * Z, n->stream);
        for (long long q = 0; q < nb && !rc && e == cudaSuccess; ++q) {
            if (graph) e = cudaGraphLaunch(graph, n->stream);
            else rc = train_step(n, B, (float)lr, eloss, true);
            if (!rc && e == cudaSuccess) n->adam_t += 1;
        }
        if (eloss && !rc && e == cudaSuccess) {
            e = cudaMemcpyAsync(lossb.data(), eloss, sizeof(double) * Z, cudaMemcpyDeviceToHost, n->stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
            double ep_loss = 0.0;
            for (double v : lossb) ep_loss += v / Z;
            loss_per_epoch[ep] = ep_loss / (double)nb;
        }
    }
    const cudaError_t e2 = cudaStreamSynchronize(n->stream);
    if (graph) cudaGraphExecDestroy(graph);
    if (rc) return rc;
    if (e == cudaSuccess) e = e2;
    if (e != cudaSuccess) return cuda_fail(e, "training");
    return check_device_error(n);
}

int it_test_refuse_recording(it_mlp *n, int on) {
    if (!n || (on != 0 && on != 1)) return mfail(IT_EINVAL, "bad argument");
    n->refuse_recording = on;
    return IT_OK;
}

int it_mlp_loss_grad(it_mlp *n, int64_t count, const double *x, const double *y, float *grads, double *loss) {
    if (!n || !x || !y || count < 1 || count > n->bmax) return mfail(IT_EINVAL, "bad argument");
    float *dX = nullptr, *dY = nullptr;
    bool own = false;
    int rc = upload_inputs(n, count, x, y, &dX, &dY, &own);
    if (rc) return rc;
    rc = gather(n, dX, dY, nullptr, 0, (int)count);
    if (!rc) rc = forward(n, (int)count, true);
    if (!rc) rc = backward(n, (int)count, n->loss, false);
    if (!rc && grads) {
        cudaError_t e = cudaMemcpyAsync(grads, n->grad, sizeof(float) * n->members * P, cudaMemcpyDeviceToHost, n->stream);
        if (e != cudaSuccess) rc = cuda_fail(e, "grad copy");
    }
    if (!rc && loss) {
        cudaError_t e = cudaMemcpyAsync(loss, n->loss, sizeof(double) * n->members, cudaMemcpyDeviceToHost, n->stream);
        if (e != cudaSuccess) rc = cuda_fail(e, "loss copy");
    }
    cudaStreamSynchronize(n->stream);
    if (own) cudaFree(dX);
    if (!rc) rc = check_device_error(n);
    return rc;
}

int it_mlp_adam_step(it_mlp *n, double lr) {
    if (!n || !(lr > 0)) return mfail(IT_EINVAL, "bad argument");
    std::vector<float2> c;
    int rc = adam_begin(n, 1, 0, c);
    if (!rc) rc = adam_step(n, (float)lr);
    if (!rc) n->adam_t += 1;
    const cudaError_t e = cudaStreamSynchronize(n->stream);   // c is released on return
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "Adam step");
    return IT_OK;
}

int it_mlp_predict(it_mlp *n, int64_t count, const double *x, double *mean, double *spread, double *per_member) {
    if (!n || !x || count < 0) return mfail(IT_EINVAL, "bad argument");
    if (count == 0) return IT_OK;
    float *dX = nullptr;
    bool own = false;
    int rc = upload_inputs(n, count, x, nullptr, &dX, nullptr, &own);
    if (rc) return rc;
    auto collect = [&](long long b0, int B, const float *fb) {   // fb: [member][B]
        for (int m = 0; m < B; ++m) {
            double s = 0, lo = 1e300, hi = -1e300;
            for (int z = 0; z < n->members; ++z) {
                const double v = fb[(size_t)z * B + m];
                s += v; lo = std::min(lo, v); hi = std::max(hi, v);
                if (per_member) per_member[(b0 + m) * n->members + z] = v;
            }
            if (mean) mean[b0 + m] = s / n->members;
            if (spread) spread[b0 + m] = hi - lo;
        }
    };
    std::vector<float> f((size_t)n->members * std::min<long long>(n->bmax, count));
    cudaError_t e = cudaSuccess;
    for (long long b0 = 0; b0 < count && !rc && e == cudaSuccess; b0 += n->bmax) {
        const int B = (int)std::min<long long>(n->bmax, count - b0);
        rc = gather(n, dX + b0 * NIN, nullptr, nullptr, 0, B);
        if (!rc) rc = forward(n, B, false);
        if (!rc) e = cudaMemcpyAsync(f.data(), n->fhat, sizeof(float) * n->members * B, cudaMemcpyDeviceToHost, n->stream);
        if (!rc && e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
        if (!rc && e == cudaSuccess) collect(b0, B, f.data());
    }
    if (!rc && e != cudaSuccess) rc = cuda_fail(e, "predict copy");
    if (rc) cudaStreamSynchronize(n->stream);
    if (own) cudaFree(dX);
    if (!rc) rc = check_device_error(n);
    return rc;
}

int it_mlp_destroy(it_mlp *n) {
    mlp_free(n);
    return IT_OK;
}

}  // extern "C"
