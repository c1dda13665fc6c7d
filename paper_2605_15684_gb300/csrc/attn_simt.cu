// attn_simt.cu -- fp32 block-sparse attention forward on CUDA cores (Sec. 2.2
// Efficient Sparse Execution; Algorithm 1 SparseAttention over the expanded mask).
//
// One CTA of 128 threads per (batch*head, query block). The kept key blocks are visited in list
// order; each block's K and V rows (gathered through the shifted grid, any shift) are staged in
// shared memory, S = Q K^T and O += P V run as register-tiled fp32 products (simt_tile.cuh), and the
// block is folded into an online softmax with expf. P takes the place of K once S is done, so three
// CTAs fit an SM (52 KB each).
// This path serves fp32 inputs, where the tensor-core path's bf16 operands would
// not meet fp32 accuracy.
#include "common.cuh"
#include "simt_tile.cuh"

namespace ssba {

namespace {

using namespace simt;

constexpr size_t kSmem = 3 * kTileFloats * sizeof(float);

__global__ void __launch_bounds__(kThreads, 3) ssba_attn_simt_f32_kernel(
    const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V, Grid g, int keep,
    float scale, const int32_t* __restrict__ idx, const int32_t* __restrict__ cnt, float* __restrict__ O,
    float* __restrict__ lse)
{
    extern __shared__ float4 raw[];
    float* Qs = reinterpret_cast<float*>(raw);
    float* Ks = Qs + kTileFloats;  // then P
    float* Vs = Ks + kTileFloats;
    const int label = blockIdx.x, bh = blockIdx.y;
    const int Tb = g.Tb();
    const int N = g.H * g.W;
    const int tx = threadIdx.x & 15;
    const float* Kh = K + (size_t)bh * N * kD;
    const float* Vh = V + (size_t)bh * N * kD;
    int qtok[kR];
    row_tokens(g, label, qtok);
    stage(Qs, Q + (size_t)bh * N * kD, qtok);

    float2 o[kR][2];
    float m[kR], l[kR];  // l: this thread's part of the row sums
#pragma unroll
    for (int a = 0; a < kR; ++a) {
        o[a][0] = o[a][1] = make_float2(0.f, 0.f);
        m[a] = -INFINITY;
        l[a] = 0.f;
    }
    const int32_t* list = idx + ((size_t)bh * Tb + label) * keep;
    const int nblk = min(max(cnt[(size_t)bh * Tb + label], 0), keep);

    for (int t = 0; t < nblk; ++t) {
        const int j = list[t];
        if ((unsigned)j >= (unsigned)Tb) continue;  // malformed label: skipped, never read out of bounds
        int tok[kR];
        row_tokens(g, j, tok);
        __syncthreads();  // the last block's P and V are consumed
        stage(Ks, Kh, tok);
        stage(Vs, Vh, tok);
        __syncthreads();
        float s[kR][4];
        dot_rows(s, Qs, Ks);
#pragma unroll
        for (int a = 0; a < kR; ++a) {
            float bmax = -INFINITY;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                s[a][b] *= scale;
                bmax = fmaxf(bmax, s[a][b]);
            }
            const float mnew = fmaxf(m[a], row_max(bmax));
            const float alpha = expf(m[a] - mnew);  // 0 on the first block (m = -inf)
            m[a] = mnew;
            l[a] *= alpha;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                s[a][b] = expf(s[a][b] - mnew);
                l[a] += s[a][b];
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                o[a][h].x *= alpha;
                o[a][h].y *= alpha;
            }
        }
        __syncthreads();  // K is consumed
        put(Ks, s);
        __syncthreads();
        add_product(o, Ks, Vs);
    }
#pragma unroll
    for (int a = 0; a < kR; ++a) {
        const float sum = row_sum(l[a]);
        const float inv = sum > 0.f ? 1.f / sum : 0.f;  // an empty list gives O = 0, lse = -inf
        const size_t row = (size_t)bh * N + qtok[a];
        *reinterpret_cast<float4*>(O + row * kD + 4 * tx) =
            make_float4(o[a][0].x * inv, o[a][0].y * inv, o[a][1].x * inv, o[a][1].y * inv);
        if (tx == 0) lse[row] = sum > 0.f ? m[a] + logf(sum) : -INFINITY;
    }
}

}  // namespace

int launch_attn_simt_f32(const ssba_desc& d, const Grid& g, int keep, float scale, const float* Q,
                         const float* K, const float* V, const int32_t* idx, const int32_t* cnt, float* O,
                         float* lse, cudaStream_t st)
{
    if (d.head_dim != kD || g.blk * g.blk != kP) {
        set_error("ssba_forward (fp32): needs head_dim=%d and block=8", kD);
        return SSBA_ERR_UNSUPPORTED;
    }
    static PerDeviceOnce attr;
    attr.run([] {
        cudaFuncSetAttribute(ssba_attn_simt_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    });
    dim3 grid(g.Tb(), d.B * d.heads);
    ssba_attn_simt_f32_kernel<<<grid, kThreads, kSmem, st>>>(Q, K, V, g, keep, scale, idx, cnt, O, lse);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("ssba_attn_simt_f32_kernel launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

}  // namespace ssba
