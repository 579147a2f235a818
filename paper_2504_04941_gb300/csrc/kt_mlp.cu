// kt_mlp.cu -- training and batch inference of the learned-guess MLP.
//
// Parameters live twice: FP32 master weights (Adam state beside them) and the packed
// BF16 block of kt_mlp.cuh that the tensor-core kernels read.  One training step:
//   train_tile    one block per 64 samples, a warp per 16: the parameters are staged in
//                 shared memory by 16-byte asynchronous copies, then forward, MSE loss gradient and backward
//                 (dz_l = (dz_{l+1} W_{l+1}) * s_l) with activations h_l and SiLU
//                 derivatives s_l / dz_l kept in shared memory as BF16, then this tile's
//                 dW_l = dz_l^T h_{l-1} and db_l into the block's own FP32 partial;
//   reduce_grads  the partials summed in block order (deterministic);
//   adam          FP32 Adam on the master weights, then the BF16 repack.
// All products are mma.sync m16n8k16 BF16 x BF16 -> FP32, operands by ldmatrix.
// What bounds it: latency (0.9 GFLOP and 0.7 MB at a batch of 4,096).  Before, a tile read
// every weight fragment from global memory, 25 single warps summed dW over the whole batch
// and 400 threads the biases one sample at a time: 657 us for loss and gradients at a batch of
// 4,096, copies to the host included; now 122 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <fstream>
#include <random>
#include <string>
#include <vector>

#include "kt_internal.h"
#include "kt_mlp.cuh"
#include "kt_tma.cuh"   // smem_u32

namespace kt {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// FP32 master parameter offsets (floats), unpadded [out][in].
struct Master {
    static constexpr int W1 = 0;                         // [128][16]
    static constexpr int W2 = W1 + kMlpH * kMlpIn;       // [128][128]
    static constexpr int W3 = W2 + kMlpH * kMlpH;
    static constexpr int W4 = W3 + kMlpH * kMlpH;        // [16][128]
    static constexpr int B1 = W4 + kMlpOut * kMlpH;
    static constexpr int B2 = B1 + kMlpH;
    static constexpr int B3 = B2 + kMlpH;
    static constexpr int B4 = B3 + kMlpH;
    static constexpr int N = B4 + kMlpOut;
};

__device__ __forceinline__ float silu_grad_f(float z)
{
    const float s = 1.0f / (1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// The packed parameters to shared memory, 16 bytes per copy.  The wait is the hardware's own and
// cannot give up, so no launch leaves its outputs unwritten.  Every thread of the block calls it.
__device__ __forceinline__ void stage_params(unsigned char *sm, const unsigned char *P)
{
    static_assert(MlpLayout::BYTES % 16 == 0, "16-byte copies");
    for (int i = threadIdx.x * 16; i < MlpLayout::BYTES; i += blockDim.x * 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(sm + i)),
                     "l"(__cvta_generic_to_global(P + i))
                     : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// 8x8 BF16 blocks of shared memory, transposed (lane 8 i + r gives row r of block i).
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const __nv_bfloat16 *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p))
                 : "memory");
}

// B fragments of two neighbouring 8-column tiles (columns c0, c0 + 8) of a row-major [k][c]
// array, reduction rows k0 .. k0 + 15: b[0], b[1] of the first tile, b[2], b[3] of the second.
__device__ __forceinline__ void b_rows(uint32_t (&b)[4], const __nv_bfloat16 *src, int ld, int k0, int c0, int lane)
{
    ldsm4t(b, src + (k0 + (lane & 7) + (lane & 8)) * ld + c0 + ((lane & 16) >> 1));
}

// A fragment (rows r0 .. r0 + 15) of the transpose of a row-major [k][r] array.
__device__ __forceinline__ void a_cols(uint32_t (&a)[4], const __nv_bfloat16 *src, int ld, int k0, int r0, int lane)
{
    ldsm4t(a, src + (k0 + (lane & 7) + ((lane & 16) >> 1)) * ld + r0 + (lane & 8));
}

// dh = dz W for W [n][k], n the reduction index (KCN chunks of 16).
template <int KCN>
__device__ __forceinline__ void back_data(const __nv_bfloat16 *W, const uint32_t (&a)[KCN][4], float (&acc)[16][4],
                                          int lane)
{
#pragma unroll
    for (int nt = 0; nt < 16; nt += 2) {
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[nt][i] = acc[nt + 1][i] = 0.0f;
#pragma unroll
        for (int kc = 0; kc < KCN; ++kc) {
            uint32_t b[4];
            b_rows(b, W, kMlpKP, kc * 16, nt * 8, lane);
            mma_bf16(acc[nt], a[kc], b[0], b[1]);
            mma_bf16(acc[nt + 1], a[kc], b[2], b[3]);
        }
    }
}

constexpr int kTile = 64;                 // samples per block
constexpr int kTrainWarps = kTile / 16;
constexpr int kMaxPartials = 512;         // blocks of one launch; each loops over its tiles

// Shared memory of train_tile (bytes): the packed parameters, the activations h0 .. h3 and
// the SiLU derivatives s1 .. s3, overwritten by dz1 .. dz3, and dz4; rows padded by 16 bytes.
struct TileLayout {
    static constexpr int H0 = MlpLayout::BYTES;
    static constexpr int H1 = H0 + kTile * kMlpKP1 * 2;
    static constexpr int HB = kTile * kMlpKP * 2;
    static constexpr int D1 = H1 + 3 * HB;
    static constexpr int D4 = D1 + 3 * HB;
    static constexpr int LOSS = D4 + kTile * kMlpKP1 * 2;
    static constexpr int BYTES = LOSS + kTrainWarps * 8;
};

struct TrainArgs {
    const unsigned char *P;          // packed bf16 parameters
    const float *X, *Tg;             // [B][16], [B][16]
    float *part;                     // [blocks][Master::N]
    double *loss;                    // [blocks]
    int B, nout;
};

__global__ void __launch_bounds__(kTrainWarps * 32, 1) train_tile(const TrainArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    stage_params(sm, a.P);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    auto rows = [&](int off) { return reinterpret_cast<__nv_bfloat16 *>(sm + off); };
    __nv_bfloat16 *H0 = rows(TileLayout::H0), *D4 = rows(TileLayout::D4);
    __nv_bfloat16 *H[3], *D[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        H[l] = rows(TileLayout::H1 + l * TileLayout::HB);
        D[l] = rows(TileLayout::D1 + l * TileLayout::HB);
    }
    const int r0 = wid * 16;   // the warp's rows of the tile
    const float invB = 1.0f / static_cast<float>(a.B);
    float *part = a.part + static_cast<size_t>(blockIdx.x) * Master::N;
    double lsum = 0.0;
    const int tiles = (a.B + kTile - 1) / kTile;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const bool first = tile == static_cast<int>(blockIdx.x);
        const long long m0 = static_cast<long long>(tile) * kTile + r0;
        // input fragment straight from X (rows beyond B are zero)
        auto xin = [&](long long m, int k) {
            const float *x = a.X + m * kMlpIn + k;   // (known to be 4-byte aligned only)
            return m < a.B ? pack_bf16(x[0], x[1]) : 0u;
        };
        uint32_t a0[1][4], ha[8][4], hb[8][4];
        a0[0][0] = xin(m0 + g, 2 * t);
        a0[0][1] = xin(m0 + g + 8, 2 * t);
        a0[0][2] = xin(m0 + g, 8 + 2 * t);
        a0[0][3] = xin(m0 + g + 8, 8 + 2 * t);
        auto put = [&](__nv_bfloat16 *dst, int ld, int c, uint32_t lo, uint32_t hi) {   // rows g, g + 8
            *reinterpret_cast<uint32_t *>(dst + (r0 + g) * ld + c) = lo;
            *reinterpret_cast<uint32_t *>(dst + (r0 + g + 8) * ld + c) = hi;
        };
        put(H0, kMlpKP1, 2 * t, a0[0][0], a0[0][1]);
        put(H0, kMlpKP1, 8 + 2 * t, a0[0][2], a0[0][3]);
        float acc[16][4];
        // SiLU derivatives and activations of one layer to shared memory
        auto keep = [&](int l, const uint32_t (&h)[8][4]) {
#pragma unroll
            for (int nt = 0; nt < 16; ++nt)
                put(D[l], kMlpKP, nt * 8 + 2 * t, pack_bf16(silu_grad_f(acc[nt][0]), silu_grad_f(acc[nt][1])),
                    pack_bf16(silu_grad_f(acc[nt][2]), silu_grad_f(acc[nt][3])));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                put(H[l], kMlpKP, 16 * j + 2 * t, h[j][0], h[j][1]);
                put(H[l], kMlpKP, 16 * j + 8 + 2 * t, h[j][2], h[j][3]);
            }
        };
        mlp_hidden<1>(sm, MlpLayout::W1, MlpLayout::B1, kMlpKP1, a0, ha, acc, lane);
        keep(0, ha);
        mlp_hidden<8>(sm, MlpLayout::W2, MlpLayout::B2, kMlpKP, ha, hb, acc, lane);
        keep(1, hb);
        mlp_hidden<8>(sm, MlpLayout::W3, MlpLayout::B3, kMlpKP, hb, ha, acc, lane);
        keep(2, ha);
        // output and loss gradient dz4 = (out - t) / B (rows beyond B and columns beyond nout: 0)
        float d[kMlpOutTiles][4];
        mlp_out(sm, ha, d, lane);
        double ls = 0.0;
#pragma unroll
        for (int nt = 0; nt < kMlpOutTiles; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const long long m = m0 + g + (i >= 2 ? 8 : 0);
                const int o = nt * 8 + 2 * t + (i & 1);
                float r = 0.0f;
                if (m < a.B && o < a.nout) r = d[nt][i] - a.Tg[m * kMlpOut + o];
                ls += 0.5 * static_cast<double>(r) * r;
                d[nt][i] = r * invB;
            }
        lsum += ls;
        uint32_t ad4[1][4];
        ad4[0][0] = pack_bf16(d[0][0], d[0][1]);
        ad4[0][1] = pack_bf16(d[0][2], d[0][3]);
        ad4[0][2] = pack_bf16(d[1][0], d[1][1]);
        ad4[0][3] = pack_bf16(d[1][2], d[1][3]);
        put(D4, kMlpKP1, 2 * t, ad4[0][0], ad4[0][1]);
        put(D4, kMlpKP1, 8 + 2 * t, ad4[0][2], ad4[0][3]);
        // backward through the layers; dz_l replaces s_l in place (each lane its own entries)
        auto times_s = [&](int l, uint32_t (&dz)[8][4]) {
#pragma unroll
            for (int nt = 0; nt < 16; ++nt) {
                uint32_t *lo = reinterpret_cast<uint32_t *>(D[l] + (r0 + g) * kMlpKP + nt * 8 + 2 * t);
                uint32_t *hi = reinterpret_cast<uint32_t *>(D[l] + (r0 + g + 8) * kMlpKP + nt * 8 + 2 * t);
                const float2 s0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(lo));
                const float2 s1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(hi));
                const uint32_t v0 = pack_bf16(acc[nt][0] * s0.x, acc[nt][1] * s0.y);
                const uint32_t v1 = pack_bf16(acc[nt][2] * s1.x, acc[nt][3] * s1.y);
                *lo = v0;
                *hi = v1;
                dz[nt >> 1][2 * (nt & 1)] = v0;
                dz[nt >> 1][2 * (nt & 1) + 1] = v1;
            }
        };
        back_data<1>(reinterpret_cast<const __nv_bfloat16 *>(sm + MlpLayout::W4), ad4, acc, lane);
        times_s(2, ha);
        back_data<8>(reinterpret_cast<const __nv_bfloat16 *>(sm + MlpLayout::W3), ha, acc, lane);
        times_s(1, hb);
        back_data<8>(reinterpret_cast<const __nv_bfloat16 *>(sm + MlpLayout::W2), hb, acc, lane);
        times_s(0, ha);
        __syncthreads();
        // dW_l = dz_l^T h_{l-1} over the tile: 16 rows at a time per warp
        auto dw = [&](const __nv_bfloat16 *Dl, int ldd, const __nv_bfloat16 *Hl, int ldh, int row, int c_lo, int c_hi,
                      float *G, int ncols) {
            uint32_t af[kTile / 16][4];
#pragma unroll
            for (int k = 0; k < kTile / 16; ++k) a_cols(af[k], Dl, ldd, 16 * k, row, lane);
            for (int c = c_lo; c < c_hi; c += 16) {
                float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < kTile / 16; ++k) {
                    uint32_t b[4];
                    b_rows(b, Hl, ldh, 16 * k, c, lane);
                    mma_bf16(s0, af[k], b[0], b[1]);
                    mma_bf16(s1, af[k], b[2], b[3]);
                }
                auto out = [&](int r, int col, float x, float y) {
                    float2 *q = reinterpret_cast<float2 *>(G + r * ncols + col);
                    float2 v = make_float2(x, y);
                    if (!first) {
                        const float2 p = *q;
                        v.x += p.x;
                        v.y += p.y;
                    }
                    *q = v;
                };
                out(row + g, c + 2 * t, s0[0], s0[1]);
                out(row + g + 8, c + 2 * t, s0[2], s0[3]);
                out(row + g, c + 8 + 2 * t, s1[0], s1[1]);
                out(row + g + 8, c + 8 + 2 * t, s1[2], s1[3]);
            }
        };
        for (int row = wid * 16; row < kMlpH; row += kTrainWarps * 16) {
            dw(D[0], kMlpKP, H0, kMlpKP1, row, 0, kMlpIn, part + Master::W1, kMlpIn);
            dw(D[1], kMlpKP, H[0], kMlpKP, row, 0, kMlpH, part + Master::W2, kMlpH);
            dw(D[2], kMlpKP, H[1], kMlpKP, row, 0, kMlpH, part + Master::W3, kMlpH);
        }
        constexpr int kc4 = kMlpH / kTrainWarps;
        dw(D4, kMlpKP1, H[2], kMlpKP, 0, wid * kc4, (wid + 1) * kc4, part + Master::W4, kMlpH);
        // db_l: one column per thread, samples in order
        for (int i = threadIdx.x; i < 3 * kMlpH + kMlpOut; i += blockDim.x) {
            const int l = i / kMlpH, n = i - l * kMlpH, ld = l < 3 ? kMlpKP : kMlpKP1;
            const __nv_bfloat16 *Dl = l < 3 ? D[0] + l * (TileLayout::HB / 2) : D4;
            float s = 0.0f;
#pragma unroll 16
            for (int m = 0; m < kTile; ++m) s += __bfloat162float(Dl[m * ld + n]);
            float *q = part + Master::B1 + i;
            *q = first ? s : *q + s;
        }
        __syncthreads();
    }
    for (int off = 16; off > 0; off >>= 1) lsum += __shfl_xor_sync(kFull, lsum, off);
    double *lw = reinterpret_cast<double *>(sm + TileLayout::LOSS);
    if (lane == 0) lw[wid] = lsum / a.B;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kTrainWarps; ++w) s += lw[w];
        a.loss[blockIdx.x] = s;
    }
}

// Partials summed in block order, eight at a time in flight; the loss by the first thread.
__global__ void __launch_bounds__(128) reduce_grads(const float *__restrict__ part, const double *__restrict__ lpart,
                                                    int blocks, float *grad, double *loss)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
    static_assert(Master::N % 4 == 0, "four gradients per thread");
    if (i < Master::N) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int b = 0; b < blocks; ++b) {
            const float4 v = *reinterpret_cast<const float4 *>(part + static_cast<size_t>(b) * Master::N + i);
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
        *reinterpret_cast<float4 *>(grad + i) = s;
    }
    if (i == 0) {
        double s = 0.0;
#pragma unroll 8
        for (int b = 0; b < blocks; ++b) s += lpart[b];
        *loss = s;
    }
}

// Adam on the FP32 masters, then refresh the packed BF16 block; rows of W1 beyond
// the input width and of W4 / b4 beyond nout stay zero.
__global__ void adam(float *p, float *m, float *v, const float *g, unsigned char *P, int step, float lr, int nin,
                     int nout)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Master::N) return;
    bool frozen = false;
    if (i < Master::W2) frozen = (i % kMlpIn) >= nin;
    else if (i >= Master::W4 && i < Master::B1) frozen = (i - Master::W4) / kMlpH >= nout;
    else if (i >= Master::B4) frozen = (i - Master::B4) >= nout;
    if (!frozen) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float mh = mi / (1.0f - powf(b1, static_cast<float>(step)));
        const float vh = vi / (1.0f - powf(b2, static_cast<float>(step)));
        p[i] -= lr * mh / (sqrtf(vh) + eps);
    }
    const float x = p[i];
    __nv_bfloat16 *Wb;
    if (i < Master::W2) {
        Wb = reinterpret_cast<__nv_bfloat16 *>(P + MlpLayout::W1) + (i / kMlpIn) * kMlpKP1 + i % kMlpIn;
        *Wb = __float2bfloat16(x);
    } else if (i < Master::W3) {
        const int j = i - Master::W2;
        reinterpret_cast<__nv_bfloat16 *>(P + MlpLayout::W2)[(j / kMlpH) * kMlpKP + j % kMlpH] = __float2bfloat16(x);
    } else if (i < Master::W4) {
        const int j = i - Master::W3;
        reinterpret_cast<__nv_bfloat16 *>(P + MlpLayout::W3)[(j / kMlpH) * kMlpKP + j % kMlpH] = __float2bfloat16(x);
    } else if (i < Master::B1) {
        const int j = i - Master::W4;
        reinterpret_cast<__nv_bfloat16 *>(P + MlpLayout::W4)[(j / kMlpH) * kMlpKP + j % kMlpH] = __float2bfloat16(x);
    } else if (i < Master::B2) {
        reinterpret_cast<float *>(P + MlpLayout::B1)[i - Master::B1] = x;
    } else if (i < Master::B3) {
        reinterpret_cast<float *>(P + MlpLayout::B2)[i - Master::B2] = x;
    } else if (i < Master::B4) {
        reinterpret_cast<float *>(P + MlpLayout::B3)[i - Master::B3] = x;
    } else {
        reinterpret_cast<float *>(P + MlpLayout::B4)[i - Master::B4] = x;
    }
}

// batch inference: X [n][16] -> out [n][16], one warp per 16 rows, the parameters staged in
// shared memory once per block (4,096 rows: 20.8 us reading them from global memory fragment by
// fragment, 16.7 now; 1,000,000 rows: 659 us, 505 now)
__global__ void __launch_bounds__(256, 2) infer(const unsigned char *P, const float *X, float *out, long long n)
{
    extern __shared__ __align__(16) unsigned char sm[];
    stage_params(sm, P);
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    for (long long m0 = ((static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * 16; m0 < n;
         m0 += static_cast<long long>(gridDim.x) * (blockDim.x / 2)) {
        auto xin = [&](long long m, int k) {
            const float *x = X + m * kMlpIn + k;   // (known to be 4-byte aligned only)
            return m < n ? pack_bf16(x[0], x[1]) : 0u;
        };
        uint32_t a0[1][4];
        a0[0][0] = xin(m0 + g, 2 * t);
        a0[0][1] = xin(m0 + g + 8, 2 * t);
        a0[0][2] = xin(m0 + g, 8 + 2 * t);
        a0[0][3] = xin(m0 + g + 8, 8 + 2 * t);
        float d[kMlpOutTiles][4];
        mlp_forward16(sm, a0, d, lane);
        const long long r0 = m0 + g, r1 = m0 + g + 8;
#pragma unroll
        for (int nt = 0; nt < kMlpOutTiles; ++nt) {
            if (r0 < n) {
                out[r0 * kMlpOut + nt * 8 + 2 * t] = d[nt][0];
                out[r0 * kMlpOut + nt * 8 + 2 * t + 1] = d[nt][1];
            }
            if (r1 < n) {
                out[r1 * kMlpOut + nt * 8 + 2 * t] = d[nt][2];
                out[r1 * kMlpOut + nt * 8 + 2 * t + 1] = d[nt][3];
            }
        }
    }
}

}  // namespace
}  // namespace kt

// ------------------------------------------------------------------ host side

namespace {

int mfail(int code, const char *msg)
{
    kt::set_error(msg);
    return code;
}

int mcuda(cudaError_t e, const char *what)
{
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    kt::set_error(m.c_str());
    return KT_ECUDA;
}

}  // namespace

struct kt_mlp {
    int nin = 0, nout = 0, device = 0;
    unsigned long long seed = 0;
    int step = 0;
    unsigned char *P = nullptr;                   // packed bf16 block (MlpLayout)
    float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;   // masters, Adam, grads
    int cap = 0;                                  // training blocks the buffers below hold
    float *part = nullptr;                        // their gradient partials [cap][Master::N]
    double *lpart = nullptr;                      // and losses [cap]
    double *loss = nullptr;                       // the batch's loss
    std::vector<float> norm = std::vector<float>(kt::MlpLayout::NNORM, 0.0f);

    ~kt_mlp()
    {
        cudaFree(P);
        cudaFree(p);
        cudaFree(m);
        cudaFree(v);
        cudaFree(g);
        cudaFree(part);
        cudaFree(lpart);
        cudaFree(loss);
    }

    int ensure(int blocks)
    {
        if (blocks <= cap) return KT_OK;
        cudaFree(part);
        cudaFree(lpart);
        part = nullptr;
        lpart = nullptr;
        cap = 0;
        cudaError_t e = cudaMalloc(&part, static_cast<size_t>(blocks) * kt::Master::N * sizeof(float));
        if (e == cudaSuccess) e = cudaMalloc(&lpart, static_cast<size_t>(blocks) * sizeof(double));
        if (e != cudaSuccess) return mfail(KT_ENOMEM, "kt_mlp: gradient partials");
        cap = blocks;
        return KT_OK;
    }

    // repack the masters into the bf16 block (adam with lr = 0 and no state change)
    int repack_all(cudaStream_t s)
    {
        std::vector<float> h(kt::Master::N);
        cudaError_t e = cudaMemcpy(h.data(), p, h.size() * 4, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return mcuda(e, "kt_mlp repack");
        std::vector<unsigned char> blk(kt::MlpLayout::BYTES, 0);
        auto putw = [&](int off, int kp, int rows, int cols, int moff) {
            for (int r = 0; r < rows; ++r)
                for (int c = 0; c < cols; ++c) {
                    __nv_bfloat16 b = __float2bfloat16(h[moff + r * cols + c]);
                    std::memcpy(blk.data() + off + 2 * (r * kp + c), &b, 2);
                }
        };
        putw(kt::MlpLayout::W1, kt::kMlpKP1, kt::kMlpH, kt::kMlpIn, kt::Master::W1);
        putw(kt::MlpLayout::W2, kt::kMlpKP, kt::kMlpH, kt::kMlpH, kt::Master::W2);
        putw(kt::MlpLayout::W3, kt::kMlpKP, kt::kMlpH, kt::kMlpH, kt::Master::W3);
        putw(kt::MlpLayout::W4, kt::kMlpKP, kt::kMlpOut, kt::kMlpH, kt::Master::W4);
        std::memcpy(blk.data() + kt::MlpLayout::B1, h.data() + kt::Master::B1, 4 * kt::kMlpH);
        std::memcpy(blk.data() + kt::MlpLayout::B2, h.data() + kt::Master::B2, 4 * kt::kMlpH);
        std::memcpy(blk.data() + kt::MlpLayout::B3, h.data() + kt::Master::B3, 4 * kt::kMlpH);
        std::memcpy(blk.data() + kt::MlpLayout::B4, h.data() + kt::Master::B4, 4 * kt::kMlpOut);
        std::memcpy(blk.data() + kt::MlpLayout::NORM, norm.data(), 4 * norm.size());
        e = cudaMemcpyAsync(P, blk.data(), blk.size(), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return mcuda(e, "kt_mlp repack upload");
        return KT_OK;
    }
};

namespace kt {
const unsigned char *mlp_device_block(const kt_mlp *m, int *nin, int *nout, int *device)
{
    if (!m) return nullptr;
    *nin = m->nin;
    *nout = m->nout;
    *device = m->device;
    return m->P;
}
}  // namespace kt

extern "C" {

int kt_mlp_sizes(int *n_master, int *packed_bytes)
{
    if (n_master) *n_master = kt::Master::N;
    if (packed_bytes) *packed_bytes = kt::MlpLayout::BYTES;
    return KT_OK;
}

int kt_mlp_create(int n_in, int n_out, unsigned long long seed, kt_mlp **out)
{
    if (!out || n_in < 1 || n_in > kt::kMlpIn || n_out < 1 || n_out > kt::kMlpOut)
        return mfail(KT_EINVAL, "kt_mlp_create: n_in must be 1..16 and n_out 1..16");
    *out = nullptr;
    kt_mlp *m = new (std::nothrow) kt_mlp();
    if (!m) return mfail(KT_ENOMEM, "kt_mlp_create: out of memory");
    m->nin = n_in;
    m->nout = n_out;
    m->seed = seed;
    cudaGetDevice(&m->device);
    cudaError_t e = cudaMalloc(&m->P, kt::MlpLayout::BYTES);
    if (e == cudaSuccess) e = cudaMalloc(&m->p, kt::Master::N * 4);
    if (e == cudaSuccess) e = cudaMalloc(&m->m, kt::Master::N * 4);
    if (e == cudaSuccess) e = cudaMalloc(&m->v, kt::Master::N * 4);
    if (e == cudaSuccess) e = cudaMalloc(&m->g, kt::Master::N * 4);
    if (e == cudaSuccess) e = cudaMalloc(&m->loss, sizeof(double));
    if (e == cudaSuccess) e = cudaMemset(m->m, 0, kt::Master::N * 4);
    if (e == cudaSuccess) e = cudaMemset(m->v, 0, kt::Master::N * 4);
    if (e != cudaSuccess) {
        delete m;
        return mfail(KT_ENOMEM, "kt_mlp_create: device allocation failed");
    }
    // PyTorch-style initialisation U(-1/sqrt(fan_in), 1/sqrt(fan_in)); padding stays 0
    std::vector<float> h(kt::Master::N, 0.0f);
    std::mt19937_64 rng(seed);
    auto fill = [&](int off, int rows, int cols, int fan_in, int vrows, int vcols) {
        const float bnd = 1.0f / std::sqrt(static_cast<float>(fan_in));
        std::uniform_real_distribution<float> U(-bnd, bnd);
        for (int r = 0; r < rows; ++r)
            for (int c = 0; c < cols; ++c) {
                const float x = U(rng);
                h[off + r * cols + c] = (r < vrows && c < vcols) ? x : 0.0f;
            }
    };
    fill(kt::Master::W1, kt::kMlpH, kt::kMlpIn, n_in, kt::kMlpH, n_in);
    fill(kt::Master::W2, kt::kMlpH, kt::kMlpH, kt::kMlpH, kt::kMlpH, kt::kMlpH);
    fill(kt::Master::W3, kt::kMlpH, kt::kMlpH, kt::kMlpH, kt::kMlpH, kt::kMlpH);
    fill(kt::Master::W4, kt::kMlpOut, kt::kMlpH, kt::kMlpH, n_out, kt::kMlpH);
    fill(kt::Master::B1, 1, kt::kMlpH, n_in, 1, kt::kMlpH);
    fill(kt::Master::B2, 1, kt::kMlpH, kt::kMlpH, 1, kt::kMlpH);
    fill(kt::Master::B3, 1, kt::kMlpH, kt::kMlpH, 1, kt::kMlpH);
    fill(kt::Master::B4, 1, kt::kMlpOut, kt::kMlpH, 1, n_out);
    for (int i = 0; i < 16; ++i) m->norm[16 + i] = 1.0f;
    for (int i = 0; i < 16; ++i) m->norm[48 + i] = 1.0f;
    e = cudaMemcpy(m->p, h.data(), h.size() * 4, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        delete m;
        return mcuda(e, "kt_mlp_create: upload");
    }
    int rc = m->repack_all(nullptr);
    if (rc) {
        delete m;
        return rc;
    }
    *out = m;
    return KT_OK;
}

void kt_mlp_free(kt_mlp *m) { delete m; }

int kt_mlp_set_norm(kt_mlp *m, const float *mu_in, const float *sd_in, const float *mu_out, const float *sd_out)
{
    if (!m || !mu_in || !sd_in || !mu_out || !sd_out) return mfail(KT_EINVAL, "kt_mlp_set_norm: NULL argument");
    for (int i = 0; i < m->nin; ++i) {
        if (!(sd_in[i] > 0)) return mfail(KT_EINVAL, "kt_mlp_set_norm: sd_in must be > 0");
        m->norm[i] = mu_in[i];
        m->norm[16 + i] = sd_in[i];
    }
    for (int i = 0; i < m->nout; ++i) {
        if (!(sd_out[i] > 0)) return mfail(KT_EINVAL, "kt_mlp_set_norm: sd_out must be > 0");
        m->norm[32 + i] = mu_out[i];
        m->norm[48 + i] = sd_out[i];
    }
    cudaError_t e = cudaMemcpy(m->P + kt::MlpLayout::NORM, m->norm.data(), 4 * m->norm.size(), cudaMemcpyHostToDevice);
    return e == cudaSuccess ? KT_OK : mcuda(e, "kt_mlp_set_norm");
}

static int fwd_bwd(kt_mlp *m, const float *X, const float *T, int B, cudaStream_t s)
{
    const int tiles = (B + kt::kTile - 1) / kt::kTile, blocks = tiles < kt::kMaxPartials ? tiles : kt::kMaxPartials;
    int rc = m->ensure(blocks);
    if (rc) return rc;
    cudaError_t e = cudaFuncSetAttribute(kt::train_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, kt::TileLayout::BYTES);
    if (e != cudaSuccess) return mcuda(e, "kt_mlp: train kernel attributes");
    const kt::TrainArgs a{m->P, X, T, m->part, m->lpart, B, m->nout};
    kt::train_tile<<<blocks, kt::kTrainWarps * 32, kt::TileLayout::BYTES, s>>>(a);
    kt::reduce_grads<<<(kt::Master::N / 4 + 127) / 128, 128, 0, s>>>(m->part, m->lpart, blocks, m->g, m->loss);
    e = cudaGetLastError();
    return e == cudaSuccess ? KT_OK : mcuda(e, "kt_mlp: train kernels");
}

int kt_mlp_train_step(kt_mlp *m, const float *X, const float *T, int B, float lr, double *loss, void *stream)
{
    if (!m || !X || !T || B < 1 || !(lr >= 0)) return mfail(KT_EINVAL, "kt_mlp_train_step: bad argument");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = fwd_bwd(m, X, T, B, s);
    if (rc) return rc;
    ++m->step;
    kt::adam<<<(kt::Master::N + 255) / 256, 256, 0, s>>>(m->p, m->m, m->v, m->g, m->P, m->step, lr, m->nin, m->nout);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mcuda(e, "kt_mlp: adam");
    if (loss) {
        e = cudaMemcpyAsync(loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return mcuda(e, "kt_mlp: loss readback");
    }
    return KT_OK;
}

int kt_mlp_gradients(kt_mlp *m, const float *X, const float *T, int B, float *grads, double *loss, void *stream)
{
    if (!m || !X || !T || B < 1 || !grads) return mfail(KT_EINVAL, "kt_mlp_gradients: bad argument");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = fwd_bwd(m, X, T, B, s);
    if (rc) return rc;
    cudaError_t e = cudaMemcpyAsync(grads, m->g, kt::Master::N * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? KT_OK : mcuda(e, "kt_mlp_gradients");
}

int kt_mlp_forward(const kt_mlp *m, const float *X, float *out, int64_t n, void *stream)
{
    if (!m || !X || !out || n < 0) return mfail(KT_EINVAL, "kt_mlp_forward: bad argument");
    if (n == 0) return KT_OK;
    // two blocks of the staged parameters fit in an SM's shared memory; beyond that the warps
    // take further rows from the parameters they hold, eight warps to a block, so that as many
    // share an SM as its registers allow (100,000 rows: 82.5 us with four warps, 54.1 with eight;
    // 16,384: 18.8)
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long most = 2LL * nsm;
    const int threads = (n + 63) / 64 <= most ? 128 : 256;
    const long long blocks = (n + threads / 2 - 1) / (threads / 2);
    const int smem = kt::MlpLayout::BYTES;
    cudaError_t e = cudaFuncSetAttribute(kt::infer, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return mcuda(e, "kt_mlp_forward");
    kt::infer<<<static_cast<unsigned>(blocks < most ? blocks : most), threads, smem, static_cast<cudaStream_t>(stream)>>>(
        m->P, X, out, n);
    e = cudaGetLastError();
    return e == cudaSuccess ? KT_OK : mcuda(e, "kt_mlp_forward");
}

int kt_mlp_get_params(const kt_mlp *m, float *master)
{
    if (!m || !master) return mfail(KT_EINVAL, "kt_mlp_get_params: NULL argument");
    cudaError_t e = cudaMemcpy(master, m->p, kt::Master::N * 4, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? KT_OK : mcuda(e, "kt_mlp_get_params");
}

int kt_mlp_set_params(kt_mlp *m, const float *master)
{
    if (!m || !master) return mfail(KT_EINVAL, "kt_mlp_set_params: NULL argument");
    cudaError_t e = cudaMemcpy(m->p, master, kt::Master::N * 4, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return mcuda(e, "kt_mlp_set_params");
    return m->repack_all(nullptr);
}

// File: "KTMLP2\0\0", int32 nin, nout, hidden, layers, uint64 seed, int32 step, dtype tag
// (1 = float32 masters), float norm[64], float masters[N].
int kt_mlp_save(const kt_mlp *m, const char *path)
{
    if (!m || !path) return mfail(KT_EINVAL, "kt_mlp_save: NULL argument");
    std::vector<float> h(kt::Master::N);
    cudaError_t e = cudaMemcpy(h.data(), m->p, h.size() * 4, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return mcuda(e, "kt_mlp_save");
    std::ofstream f(path, std::ios::binary);
    if (!f) return mfail(KT_EINVAL, "kt_mlp_save: cannot open file");
    const char magic[8] = {'K', 'T', 'M', 'L', 'P', '2', 0, 0};
    const int32_t hdr[4] = {m->nin, m->nout, kt::kMlpH, 4};
    const int32_t tail[2] = {m->step, 1};
    f.write(magic, 8);
    f.write(reinterpret_cast<const char *>(hdr), sizeof hdr);
    f.write(reinterpret_cast<const char *>(&m->seed), 8);
    f.write(reinterpret_cast<const char *>(tail), sizeof tail);
    f.write(reinterpret_cast<const char *>(m->norm.data()), m->norm.size() * 4);
    f.write(reinterpret_cast<const char *>(h.data()), h.size() * 4);
    return f ? KT_OK : mfail(KT_EINVAL, "kt_mlp_save: write failed");
}

int kt_mlp_load_file(const char *path, kt_mlp **out)
{
    if (!path || !out) return mfail(KT_EINVAL, "kt_mlp_load_file: NULL argument");
    *out = nullptr;
    std::ifstream f(path, std::ios::binary);
    if (!f) return mfail(KT_EINVAL, "kt_mlp_load_file: cannot open file");
    char magic[8];
    int32_t hdr[4], tail[2];
    unsigned long long seed = 0;
    std::vector<float> norm(kt::MlpLayout::NNORM), h(kt::Master::N);
    f.read(magic, 8);
    f.read(reinterpret_cast<char *>(hdr), sizeof hdr);
    f.read(reinterpret_cast<char *>(&seed), 8);
    f.read(reinterpret_cast<char *>(tail), sizeof tail);
    f.read(reinterpret_cast<char *>(norm.data()), norm.size() * 4);
    f.read(reinterpret_cast<char *>(h.data()), h.size() * 4);
    if (!f || std::memcmp(magic, "KTMLP2", 6) != 0 || hdr[2] != kt::kMlpH || hdr[3] != 4 || tail[1] != 1)
        return mfail(KT_EPARSE, "kt_mlp_load_file: not a KTMLP2 file of this architecture");
    kt_mlp *m = nullptr;
    int rc = kt_mlp_create(hdr[0], hdr[1], seed, &m);
    if (rc) return rc;
    m->step = tail[0];
    m->norm = norm;
    rc = kt_mlp_set_params(m, h.data());
    if (rc) {
        delete m;
        return rc;
    }
    *out = m;
    return KT_OK;
}

}  // extern "C"
