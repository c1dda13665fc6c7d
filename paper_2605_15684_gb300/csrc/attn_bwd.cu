// attn_bwd.cu -- gradients of the block-sparse attention (the backward pass of Algorithm 1's
// SparseAttention over the same kept blocks), on CUDA cores in fp32.
//
// For the output gradient dO, with p_nm = exp(scale q_n.k_m - lse_n) over the allowed pairs:
//   D_n  = dO_n . O_n
//   dV_m = sum_n p_nm dO_n
//   ds_nm = p_nm (dO_n . v_m - D_n)
//   dQ_n = scale sum_m ds_nm k_m,   dK_m = scale sum_n ds_nm q_n.
// Two kernels, no atomics, deterministic, 128 threads a CTA, every product a register-tiled fp32 one
// of 64 x 64 tiles in shared memory (simt_tile.cuh):
//   ssba_bwd_dq_kernel    one CTA per (batch*head, query block): the kept key blocks staged in list
//                         order; S = Q K^T, dP = dO V^T, dQ += dS K. dS takes the place of V, so
//                         three CTAs fit an SM (70 KB each). Writes dQ and D.
//   ssba_bwd_dkdv_kernel  one CTA per (batch*head, key block): finds, in ascending order, the
//                         query blocks whose lists hold it, stages each one's Q and dO, and forms
//                         S^T = K Q^T, dP^T = V dO^T, dV += P^T dO, dK += dS^T Q (P^T, then dS^T, in
//                         one tile; two CTAs an SM, 87 KB each).
#include "common.cuh"
#include "simt_tile.cuh"

namespace ssba {

namespace {

using namespace simt;

constexpr size_t kDqSmem = 4 * kTileFloats * sizeof(float);
constexpr size_t kDkvSmem = 5 * kTileFloats * sizeof(float);

template <typename T>
__global__ void __launch_bounds__(kThreads, 3) ssba_bwd_dq_kernel(
    const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V, const T* __restrict__ O,
    const float* __restrict__ lse, const T* __restrict__ dO, Grid g, int keep, float scale,
    const int32_t* __restrict__ idx, const int32_t* __restrict__ cnt, float* __restrict__ dQ,
    float* __restrict__ Dbuf)
{
    extern __shared__ float4 raw[];
    float* Qs = reinterpret_cast<float*>(raw);
    float* Gs = Qs + kTileFloats;
    float* Ks = Gs + kTileFloats;
    float* Vs = Ks + kTileFloats;  // then dS
    const int label = blockIdx.x, bh = blockIdx.y;
    const int Tb = g.Tb();
    const int N = g.H * g.W;
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    const size_t head = (size_t)bh * N * kD;
    int qtok[kR];
    row_tokens(g, label, qtok);
    stage(Qs, Q + head, qtok);
    stage(Gs, dO + head, qtok);
    __syncthreads();
    float D[kR], L[kR];
    float2 dq[kR][2];
#pragma unroll
    for (int a = 0; a < kR; ++a) {
        const size_t row = (size_t)bh * N + qtok[a];
        const float4 o = load4(O + row * kD + 4 * tx);
        const float4 go = *reinterpret_cast<const float4*>(Gs + (ty + 8 * a) * kLd + 4 * tx);
        D[a] = row_sum(fmaf(go.x, o.x, go.y * o.y) + fmaf(go.z, o.z, go.w * o.w));
        L[a] = lse[row];
        dq[a][0] = dq[a][1] = make_float2(0.f, 0.f);
        if (tx == 0) Dbuf[row] = D[a];
    }
    const int32_t* list = idx + ((size_t)bh * Tb + label) * keep;
    const int nblk = min(max(cnt[(size_t)bh * Tb + label], 0), keep);
    for (int t = 0; t < nblk; ++t) {
        const int j = list[t];
        if ((unsigned)j >= (unsigned)Tb) continue;  // malformed label: skipped, never read out of bounds
        int tok[kR];
        row_tokens(g, j, tok);
        __syncthreads();  // the last block's K and dS are consumed
        stage(Ks, K + head, tok);
        stage(Vs, V + head, tok);
        __syncthreads();
        float s[kR][4], dp[kR][4];
        dot_rows(s, Qs, Ks);
        dot_rows(dp, Gs, Vs);
#pragma unroll
        for (int a = 0; a < kR; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float pr = expf(s[a][b] * scale - L[a]);
                s[a][b] = pr * (dp[a][b] - D[a]) * scale;
            }
        __syncthreads();  // V is consumed
        put(Vs, s);
        __syncthreads();
        add_product(dq, Vs, Ks);
    }
#pragma unroll
    for (int a = 0; a < kR; ++a)
        *reinterpret_cast<float4*>(dQ + ((size_t)bh * N + qtok[a]) * kD + 4 * tx) =
            make_float4(dq[a][0].x, dq[a][0].y, dq[a][1].x, dq[a][1].y);
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 2) ssba_bwd_dkdv_kernel(
    const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V, const float* __restrict__ lse,
    const T* __restrict__ dO, const float* __restrict__ Dbuf, Grid g, int keep, float scale,
    const int32_t* __restrict__ idx, const int32_t* __restrict__ cnt, float* __restrict__ dK,
    float* __restrict__ dV)
{
    extern __shared__ float4 raw[];
    float* Ks = reinterpret_cast<float*>(raw);
    float* Vs = Ks + kTileFloats;
    float* Qs = Vs + kTileFloats;
    float* Gs = Qs + kTileFloats;
    float* Ps = Gs + kTileFloats;  // P^T, then dS^T
    __shared__ float Ls[kP], Ds[kP];
    __shared__ int qlist[kThreads];
    __shared__ int wcount[kThreads / 32];
    const int label = blockIdx.x, bh = blockIdx.y;
    const int Tb = g.Tb();
    const int N = g.H * g.W;
    const int tx = threadIdx.x & 15;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t head = (size_t)bh * N * kD;
    int ktok[kR];
    row_tokens(g, label, ktok);
    stage(Ks, K + head, ktok);
    stage(Vs, V + head, ktok);
    float2 dk[kR][2], dv[kR][2];
#pragma unroll
    for (int a = 0; a < kR; ++a) dk[a][0] = dk[a][1] = dv[a][0] = dv[a][1] = make_float2(0.f, 0.f);
    // query blocks whose lists hold this key block, in ascending order, kThreads at a time
    for (int i0 = 0; i0 < Tb; i0 += kThreads) {
        const int i = i0 + threadIdx.x;
        bool has = false;
        if (i < Tb) {
            const int32_t* list = idx + ((size_t)bh * Tb + i) * keep;
            const int n = min(max(cnt[(size_t)bh * Tb + i], 0), keep);
            for (int t = 0; t < n; ++t) has |= list[t] == label;
        }
        const unsigned b = __ballot_sync(0xffffffffu, has);
        __syncthreads();  // qlist / wcount of the previous round are consumed
        if (lane == 0) wcount[warp] = __popc(b);
        __syncthreads();
        int off = 0;
        for (int w = 0; w < warp; ++w) off += wcount[w];
        if (has) qlist[off + __popc(b & ((1u << lane) - 1u))] = i;
        int total = 0;
        for (int w = 0; w < kThreads / 32; ++w) total += wcount[w];
        __syncthreads();
        for (int u = 0; u < total; ++u) {
            const int qi = qlist[u];
            int tok[kR];
            row_tokens(g, qi, tok);
            __syncthreads();  // the last block's tiles are consumed
            stage(Qs, Q + head, tok);
            stage(Gs, dO + head, tok);
            if (threadIdx.x < kP) {
                const size_t qrow = (size_t)bh * N + g.token(qi, threadIdx.x);
                Ls[threadIdx.x] = lse[qrow];
                Ds[threadIdx.x] = Dbuf[qrow];
            }
            __syncthreads();
            float s[kR][4];
            dot_rows(s, Ks, Qs);
#pragma unroll
            for (int a = 0; a < kR; ++a)
#pragma unroll
                for (int b2 = 0; b2 < 4; ++b2) s[a][b2] = expf(s[a][b2] * scale - Ls[tx + 16 * b2]);
            put(Ps, s);
            __syncthreads();
            add_product(dv, Ps, Gs);
            float dp[kR][4];
            dot_rows(dp, Vs, Gs);
#pragma unroll
            for (int a = 0; a < kR; ++a)
#pragma unroll
                for (int b2 = 0; b2 < 4; ++b2) s[a][b2] = s[a][b2] * (dp[a][b2] - Ds[tx + 16 * b2]) * scale;
            __syncthreads();  // P^T is consumed
            put(Ps, s);
            __syncthreads();
            add_product(dk, Ps, Qs);
        }
    }
#pragma unroll
    for (int a = 0; a < kR; ++a) {
        const size_t row = ((size_t)bh * N + ktok[a]) * kD + 4 * tx;
        *reinterpret_cast<float4*>(dK + row) = make_float4(dk[a][0].x, dk[a][0].y, dk[a][1].x, dk[a][1].y);
        *reinterpret_cast<float4*>(dV + row) = make_float4(dv[a][0].x, dv[a][0].y, dv[a][1].x, dv[a][1].y);
    }
}

template <typename T>
int launch_bwd_t(const ssba_desc& d, const Grid& g, int keep, float scale, const void* Q, const void* K,
                 const void* V, const void* O, const float* lse, const void* dO, const int32_t* idx,
                 const int32_t* cnt, float* dQ, float* dK, float* dV, float* Dbuf, cudaStream_t st)
{
    static PerDeviceOnce attr;  // one for each T
    attr.run([] {
        cudaFuncSetAttribute(ssba_bwd_dq_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDqSmem);
        cudaFuncSetAttribute(ssba_bwd_dkdv_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDkvSmem);
    });
    dim3 grid(g.Tb(), d.B * d.heads);
    ssba_bwd_dq_kernel<T><<<grid, kThreads, kDqSmem, st>>>(
        static_cast<const T*>(Q), static_cast<const T*>(K), static_cast<const T*>(V), static_cast<const T*>(O), lse,
        static_cast<const T*>(dO), g, keep, scale, idx, cnt, dQ, Dbuf);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        ssba_bwd_dkdv_kernel<T><<<grid, kThreads, kDkvSmem, st>>>(
            static_cast<const T*>(Q), static_cast<const T*>(K), static_cast<const T*>(V), lse,
            static_cast<const T*>(dO), Dbuf, g, keep, scale, idx, cnt, dK, dV);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error("ssba_backward launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

}  // namespace

int launch_backward(const ssba_desc& d, const Grid& g, int keep, float scale, const void* Q, const void* K,
                    const void* V, const void* O, const float* lse, const void* dO, const int32_t* idx,
                    const int32_t* cnt, float* dQ, float* dK, float* dV, float* Dbuf, cudaStream_t st)
{
    if (d.head_dim != kD || g.blk * g.blk != kP) {
        set_error("ssba_backward: needs head_dim=%d and block=8", kD);
        return SSBA_ERR_UNSUPPORTED;
    }
    if (d.dtype == SSBA_BF16) {
        int rc = launch_backward_ws(d, g, keep, scale, Q, K, V, O, lse, dO, idx, cnt, dQ, dK, dV, Dbuf, st);
        if (rc != SSBA_ERR_UNSUPPORTED) return rc;
        rc = launch_backward_tc(d, g, keep, scale, Q, K, V, O, lse, dO, idx, cnt, dQ, dK, dV, Dbuf, st);
        if (rc != SSBA_ERR_UNSUPPORTED) return rc;
        return launch_bwd_t<__nv_bfloat16>(d, g, keep, scale, Q, K, V, O, lse, dO, idx, cnt, dQ, dK, dV, Dbuf, st);
    }
    return launch_bwd_t<float>(d, g, keep, scale, Q, K, V, O, lse, dO, idx, cnt, dQ, dK, dV, Dbuf, st);
}

}  // namespace ssba
