// simt_tile.cuh -- 64 x 64 x 64 products on the CUDA cores in fp32, for the paths whose precision the
// tensor cores' operand types would not meet (attn_simt.cu, attn_bwd.cu). 128 threads; thread
// (ty, tx) = (t / 16, t % 16) owns rows ty + 8 a of a 64 x 64 result, and of them either the columns
// tx + 16 b (a product of two tiles by rows, over head_dim) or the columns 4 tx .. 4 tx + 3 (a tile
// times a tile by columns). Tiles lie in shared memory by rows of kLd = 68 floats: the 16-byte
// chunks of 8 consecutive rows then cover all 32 banks. A thread reads 12 16-byte chunks, 8 of them
// broadcasts, for 128 multiply-adds in both products (the kernels before read one 4-byte word a
// multiply-add, two threads a row, and were bound by those reads; 4 x 4 results a thread, 8 chunks
// for 64, still were), and the multiply-adds go out as packed pairs. Measured, 24 heads: a 1024 px fp32
// layer (11 of 64 blocks) forward 1090 -> 437 us (40 TFLOP/s), gradients 2871 -> 1459 us; 512 px (3 of
// 16) 92 -> 41 and 303 -> 156 us. What is left: four barriers a block pair, and loads of the next
// tiles that only the SM's other CTAs cover.
#pragma once

#include "common.cuh"

namespace ssba {
namespace simt {

constexpr int kD = 64;         // head_dim
constexpr int kP = 64;         // tokens per block (8 x 8)
constexpr int kThreads = 128;
constexpr int kR = 8;          // rows of a thread
constexpr int kLd = 68;        // floats of a tile row in shared memory
constexpr int kTileFloats = kP * kLd;

__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p)
{
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

// Tokens of the rows ty + 8 i of block `label` (the map of Grid::token for 8x8 blocks).
__device__ __forceinline__ void row_tokens(const Grid& g, int label, int (&tok)[kR])
{
    const int br = label / g.bw, bc = label - br * g.bw;
    int c = bc * 8 + (threadIdx.x >> 4) - g.sc;  // row ty + 8 i: window row i, window column ty
    c += c < 0 ? g.W : 0;
#pragma unroll
    for (int i = 0; i < kR; ++i) {
        int r = br * 8 + i - g.sr;
        r += r < 0 ? g.H : 0;
        tok[i] = r * g.W + c;
    }
}

// Rows of block `label` of one head X [N][64] into the tile dst, as fp32 (all loads in flight first).
template <typename T>
__device__ __forceinline__ void stage(float* dst, const T* X, const int (&tok)[kR])
{
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    float4 v[kR];
#pragma unroll
    for (int i = 0; i < kR; ++i) v[i] = load4(X + (size_t)tok[i] * kD + 4 * tx);
#pragma unroll
    for (int i = 0; i < kR; ++i) *reinterpret_cast<float4*>(dst + (ty + 8 * i) * kLd + 4 * tx) = v[i];
}

// c[a][b] = sum_d A[ty + 8 a][d] B[tx + 16 b][d]: even and odd d in the two parts of a packed pair,
// added at the end.
__device__ __forceinline__ void dot_rows(float (&c)[kR][4], const float* A, const float* B)
{
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    float2 s[kR][4];
#pragma unroll
    for (int a = 0; a < kR; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) s[a][b] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int d = 0; d < kD; d += 4) {
        float4 x[kR], y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = *reinterpret_cast<const float4*>(B + (tx + 16 * i) * kLd + d);
#pragma unroll
        for (int i = 0; i < kR; ++i) x[i] = *reinterpret_cast<const float4*>(A + (ty + 8 * i) * kLd + d);
#pragma unroll
        for (int a = 0; a < kR; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                s[a][b] = __ffma2_rn(make_float2(x[a].x, x[a].y), make_float2(y[b].x, y[b].y), s[a][b]);
                s[a][b] = __ffma2_rn(make_float2(x[a].z, x[a].w), make_float2(y[b].z, y[b].w), s[a][b]);
            }
    }
#pragma unroll
    for (int a = 0; a < kR; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) c[a][b] = s[a][b].x + s[a][b].y;
}

// c[a] (columns 4 tx ..) += sum_j A[ty + 8 a][j] B[j][4 tx ..].
__device__ __forceinline__ void add_product(float2 (&c)[kR][2], const float* A, const float* B)
{
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll 2
    for (int j = 0; j < kP; j += 4) {
        float4 x[kR];
#pragma unroll
        for (int i = 0; i < kR; ++i) x[i] = *reinterpret_cast<const float4*>(A + (ty + 8 * i) * kLd + j);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 y = *reinterpret_cast<const float4*>(B + (j + k) * kLd + 4 * tx);
#pragma unroll
            for (int a = 0; a < kR; ++a) {
                const float w = k == 0 ? x[a].x : (k == 1 ? x[a].y : (k == 2 ? x[a].z : x[a].w));
                c[a][0] = __ffma2_rn(make_float2(w, w), make_float2(y.x, y.y), c[a][0]);
                c[a][1] = __ffma2_rn(make_float2(w, w), make_float2(y.z, y.w), c[a][1]);
            }
        }
    }
}

// The thread's values of a result by columns tx + 16 b, into a tile by rows.
__device__ __forceinline__ void put(float* dst, const float (&c)[kR][4])
{
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
    for (int a = 0; a < kR; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) dst[(ty + 8 * a) * kLd + tx + 16 * b] = c[a][b];
}

// Over the 16 threads of a row.
__device__ __forceinline__ float row_max(float v)
{
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float row_sum(float v)
{
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace simt
}  // namespace ssba
