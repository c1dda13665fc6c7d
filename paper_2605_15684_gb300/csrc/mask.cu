// mask.cu -- block compression, affinity and Top-k gating (Sec. 2.2; Algorithm 1,
// partition .. Top-k Smallest) as two HBM-friendly kernels:
//
//   ssba_pool_kernel    one CTA per (batch*head, block): gathers the block's 64 shifted
//                       tokens of Q and K with 16-byte loads, and writes the fp32 block
//                       means q_b, k_b (Eq. for q_b/k_b) to the workspace. Dominant cost:
//                       reading Q and K once (algorithmic bytes 2 * B * heads * N *
//                       head_dim * elem); HBM-bound.
//   ssba_select64_kernel  (head_dim 64; ssba_select_kernel for other widths) S rows = q_b[i] . k_b[j]
//                       for all j in fp32, then an exact selection of the `keep` largest entries
//                       under the total order (S descending, label ascending), i.e. the k_drop
//                       smallest are dropped and ties keep the lower label; the kept labels
//                       are written in ascending order.
//   ssba_mask_fused_kernel  both steps in one launch for head_dim 64, 8x8 blocks and at
//                       most 128 blocks: a cluster of 8 CTAs per (batch, head) pools its
//                       blocks into shared memory, reads the head's k_b from the other CTAs
//                       of the cluster (distributed shared memory), and selects its rows
//                       (keys in registers, the radix walk of sel::ballot_select). No
//                       q_b/k_b round trip through global memory and no second launch.
#include <cooperative_groups.h>
#include <cstdio>
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"
#include "select.cuh"

namespace ssba {

namespace {


template <typename T>
struct Vec;
template <>
struct Vec<__nv_bfloat16> {
    static constexpr int kElems = 8;  // 16 bytes
    __device__ static void to_f32(const uint4& v, float* out)
    {
        const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float2 f = __bfloat1622float2(p[i]);
            out[2 * i] = f.x;
            out[2 * i + 1] = f.y;
        }
    }
};
template <>
struct Vec<float> {
    static constexpr int kElems = 4;
    __device__ static void to_f32(const uint4& v, float* out)
    {
        out[0] = __uint_as_float(v.x);
        out[1] = __uint_as_float(v.y);
        out[2] = __uint_as_float(v.z);
        out[3] = __uint_as_float(v.w);
    }
};

// One CTA per (batch*head, block) for head_dim = 64, 256 threads: warp w reads tensor
// (w / 4 ? K : Q), rows [16 * (w % 4), +16) of the block. Lane l covers 16-byte chunk
// (l % 8) of rows l/8 + 4i, i < 4: four independent 16-byte loads per lane, so the whole
// block is requested in one round. Partial sums are combined in a fixed order (lanes by
// shuffles, warps through shared memory), then the block means are written.
template <typename T>
__global__ void __launch_bounds__(256) ssba_pool_kernel(const T* __restrict__ Q, const T* __restrict__ K, Grid g,
                                                        float* __restrict__ qb, float* __restrict__ kb)
{
    constexpr int kD = 64;
    constexpr int VE = Vec<T>::kElems;
    constexpr int CPR = kD / VE;            // 16-byte chunks per token row (8 bf16 / 16 fp32)
    constexpr int RPI = 32 / CPR;           // rows per warp instruction
    constexpr int ROWS = 16;                // rows per warp
    constexpr int LOADS = ROWS / RPI;       // loads per lane
    __shared__ float part[2][4][kD];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int which = warp >> 2, quarter = warp & 3;
    const int label = blockIdx.x, bh = blockIdx.y;
    const int N = g.H * g.W;
    const T* X = (which ? K : Q) + (size_t)bh * N * kD;
    const int col = lane % CPR, r0 = lane / CPR;
    uint4 v[LOADS];
#pragma unroll
    for (int i = 0; i < LOADS; ++i) {
        const int pos = quarter * ROWS + r0 + i * RPI;
        v[i] = __ldg(reinterpret_cast<const uint4*>(X + (size_t)g.token(label, pos) * kD + col * VE));
    }
    float acc[VE];
#pragma unroll
    for (int e = 0; e < VE; ++e) acc[e] = 0.f;
#pragma unroll
    for (int i = 0; i < LOADS; ++i) {
        float f[VE];
        Vec<T>::to_f32(v[i], f);
#pragma unroll
        for (int e = 0; e < VE; ++e) acc[e] += f[e];
    }
#pragma unroll
    for (int o = CPR; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < VE; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    if (r0 == 0)
#pragma unroll
        for (int e = 0; e < VE; ++e) part[which][quarter][col * VE + e] = acc[e];
    __syncthreads();
    if (threadIdx.x < 2 * kD) {
        const int w = threadIdx.x >> 6, c = threadIdx.x & (kD - 1);
        const float sum = (part[w][0][c] + part[w][1][c]) + (part[w][2][c] + part[w][3][c]);
        (w ? kb : qb)[((size_t)bh * g.Tb() + label) * kD + c] = sum * (1.0f / 64.0f);
    }
}

// Generic-width fallback (any head_dim multiple of 16 bytes): the block's tokens are
// staged in fp32 in shared memory and column sums taken in in-block position order.
template <typename T>
__global__ void __launch_bounds__(128) ssba_pool_generic_kernel(const T* __restrict__ Q, const T* __restrict__ K,
                                                                Grid g, int d, float* __restrict__ qb,
                                                                float* __restrict__ kb)
{
    extern __shared__ float stage[];  // [2][P][d]
    const int label = blockIdx.x;
    const int bh = blockIdx.y;
    const int P = g.blk * g.blk;
    const int N = g.H * g.W;
    constexpr int VE = Vec<T>::kElems;
    const int cpr = d / VE;
    const int chunks = P * cpr;
    const T* Qh = Q + (size_t)bh * N * d;
    const T* Kh = K + (size_t)bh * N * d;
    for (int ci = threadIdx.x; ci < 2 * chunks; ci += 128) {
        int which = ci >= chunks;
        int cc = which ? ci - chunks : ci;
        int pos = cc / cpr, c = cc - pos * cpr;
        int tok = g.token(label, pos);
        uint4 v = __ldg(reinterpret_cast<const uint4*>((which ? Kh : Qh) + (size_t)tok * d + c * VE));
        float f[VE];
        Vec<T>::to_f32(v, f);
        float* dst = stage + ((size_t)which * P + pos) * d + c * VE;
#pragma unroll
        for (int e = 0; e < VE; ++e) dst[e] = f[e];
    }
    __syncthreads();
    const float inv = 1.0f / (float)P;
    for (int t = threadIdx.x; t < 2 * d; t += 128) {
        int which = t >= d;
        int c = which ? t - d : t;
        const float* src = stage + (size_t)which * P * d + c;
        float acc = 0.f;
        for (int pos = 0; pos < P; ++pos) acc += src[(size_t)pos * d];
        (which ? kb : qb)[((size_t)bh * g.Tb() + label) * d + c] = acc * inv;
    }
}

constexpr int kSelWarps = 8;
constexpr int kSelKeyChunk = 256;
constexpr int kMaxTb = 2048;
constexpr size_t kSelSmem = 220 * 1024;   // largest working set of ssba_select_kernel
constexpr size_t kPoolSmem = 200 * 1024;  // of ssba_pool_generic_kernel
constexpr int kMaxGridY = 65535;  // (batch, head) pairs of a launch; more take several

// Gating of `rows` rows of keys in shared memory (row r at S + r * Tb); kept labels of row r to
// dst + r * keep.
template <int kPer>
__device__ __forceinline__ void select_rows(const uint32_t* S, int Tb, int keep, int lane, int32_t* dst, int rows)
{
    for (int r = 0; r < rows; ++r) {
        uint32_t key[kPer];
#pragma unroll
        for (int m = 0; m < kPer; ++m) {
            const int j = lane + 32 * m;
            key[m] = j < Tb ? S[(size_t)r * Tb + j] : 0u;
        }
        sel::ballot_select<kPer>(key, Tb, keep, lane, dst + (size_t)r * keep);
    }
}

// Affinity and gating for head_dim 64: a CTA takes kSelWarps * kRows rows of one head, warp w the rows
// [w kRows, (w + 1) kRows) of them; the keys' means pass through shared memory 128 at a time (rows of
// 68 floats: 8 consecutive rows cover the banks), a lane scores 4 keys (2 or 1 of the last few) against
// its warp's kRows rows at a time, and the walks (ballot_select, kPer keys a lane; 8: 2 up to 64 blocks) read the
// finished rows of keys back from shared memory. One instantiation for each register layout of the walk, so that
// the long rows' registers (64 keys a lane) do not cost the short ones theirs, and CTAs.
// What bounds it: the latency of the gating's counts (36 of 53 us at 510 blocks) and the shared-memory
// reads of the scores, 4 + kRows 16-byte chunks for 16 kRows multiply-adds of a lane. (One key at a time:
// 510 blocks 62 us, 324 39.7, 256 24.0, 64 at batch 4 9.3; now 53, 35, 20 and 9.) The kernel before (one
// row a warp, keys transposed one word at a time, a 32-bit radix walk over shared memory): 510 blocks
// 195, 256 99, 64 at batch 4 15.
constexpr int kSel64Keys = 128, kSel64Ld = 68;
// CTAs an SM that the registers leave room for: as many as run without spills.
constexpr int sel64_ctas(int rows, int per) { return per == 64 ? 1 : (rows == 4 || per == 32 ? 2 : (rows == 2 ? 3 : 4)); }
constexpr size_t sel64_smem(int rows, int Tb)
{
    return ((size_t)kSel64Keys * kSel64Ld + (size_t)kSelWarps * rows * (64 + Tb)) * sizeof(float);
}
template <int kRows, int kPer>
__global__ void __launch_bounds__(kSelWarps * 32, sel64_ctas(kRows, kPer)) ssba_select64_kernel(const float* __restrict__ qb,
                                                                       const float* __restrict__ kb, int Tb, int keep,
                                                                       int32_t* __restrict__ idx,
                                                                       int32_t* __restrict__ cnt,
                                                                       float* __restrict__ scores)
{
    constexpr int kD = 64, kCta = kSelWarps * kRows, kPerLane = kSel64Keys / 32;
    extern __shared__ float4 raw[];
    float* ks = reinterpret_cast<float*>(raw);
    float* qs = ks + kSel64Keys * kSel64Ld;                     // [kCta][64]
    uint32_t* S = reinterpret_cast<uint32_t*>(qs + kCta * kD);  // [kCta][Tb]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, bh = blockIdx.y;
    const int row0 = blockIdx.x * kCta + warp * kRows, rows = min(max(Tb - row0, 0), kRows);
    const float4* kbh = reinterpret_cast<const float4*>(kb + (size_t)bh * Tb * kD);
    ptx::grid_dep_wait();  // the means may come from the grid launched just before this one
    ptx::grid_dep_launch();
    // rows past Tb are zeros; a warp reads only its own rows
    for (int e = lane; e < kRows * (kD / 4); e += 32)
        reinterpret_cast<float4*>(qs + warp * kRows * kD)[e] =
            e / (kD / 4) < rows ? __ldg(reinterpret_cast<const float4*>(qb + ((size_t)bh * Tb + row0) * kD) + e)
                                : make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t* Sw = S + (size_t)warp * kRows * Tb;
    for (int j0 = 0; j0 < Tb; j0 += kSel64Keys) {
        const int nk = min(kSel64Keys, Tb - j0);
        __syncthreads();  // the last keys are consumed
#pragma unroll
        for (int i = 0; i < kSel64Keys * (kD / 4) / (kSelWarps * 32); ++i) {
            const int e = threadIdx.x + i * kSelWarps * 32, j = e / (kD / 4), c = e % (kD / 4);
            if (j < nk) *reinterpret_cast<float4*>(ks + j * kSel64Ld + 4 * c) = __ldg(kbh + (size_t)(j0 + j) * (kD / 4) + c);
        }
        __syncthreads();
        auto score = [&](auto n) {  // decltype(n)::value keys of a lane at a time; those past nk are not used
            constexpr int kKeys = decltype(n)::value;
#pragma unroll
            for (int m0 = 0; m0 < kPerLane; m0 += kKeys) {
                if (32 * m0 >= nk) break;
                float acc[kKeys][kRows];
                sel::affinity_keys<kRows, kKeys>(acc, qs + warp * kRows * kD, kD, [&](int k, int c) {
                    return *reinterpret_cast<const float4*>(ks + (lane + 32 * (m0 + k)) * kSel64Ld + 4 * c);
                });
#pragma unroll
                for (int k = 0; k < kKeys; ++k) {
                    const int j = lane + 32 * (m0 + k);
#pragma unroll
                    for (int r = 0; r < kRows; ++r) {
                        if (r >= rows || j >= nk) break;
                        Sw[(size_t)r * Tb + j0 + j] = sel::order_key(acc[k][r]);
                        if (scores) scores[((size_t)bh * Tb + row0 + r) * Tb + j0 + j] = acc[k][r];
                    }
                }
            }
        };
        if (kRows > 1 && nk > kSel64Keys / 2)
            score(std::integral_constant<int, 4>{});
        else if (nk > 32)
            score(std::integral_constant<int, 2>{});
        else
            score(std::integral_constant<int, 1>{});
    }
    __syncwarp();
    int32_t* dst = idx + ((size_t)bh * Tb + row0) * keep;
    if (kPer == 8 && Tb <= 64) select_rows<2>(Sw, Tb, keep, lane, dst, rows);
    else select_rows<kPer>(Sw, Tb, keep, lane, dst, rows);
    if (lane < rows) cnt[(size_t)bh * Tb + row0 + lane] = keep;
}

// One warp per query block (row i of S), kSelWarps rows per CTA.
// smem: kbT [d][kSelKeyChunk + 1] (padded transpose of a key chunk) | q rows [kSelWarps][d]
//       | S rows as order keys [kSelWarps][Tb]
// S[i][j] = q_b[i] . k_b[j] in fp32 (FMA over d in order); the row is then reduced to its
// `keep` largest entries under (S descending, label ascending), kept labels ascending.
__global__ void __launch_bounds__(kSelWarps * 32) ssba_select_kernel(const float* __restrict__ qb,
                                                                     const float* __restrict__ kb, int Tb,
                                                                     int d, int keep,
                                                                     int32_t* __restrict__ idx,
                                                                     int32_t* __restrict__ cnt,
                                                                     float* __restrict__ scores)
{
    extern __shared__ float sm[];
    constexpr int kLd = kSelKeyChunk + 1;
    float* kbT = sm;
    float* qs = kbT + (size_t)d * kLd;
    uint32_t* Skey = reinterpret_cast<uint32_t*>(qs + (size_t)kSelWarps * d);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bh = blockIdx.y;
    const int row = blockIdx.x * kSelWarps + warp;
    const bool active = row < Tb;
    const float* kbh = kb + (size_t)bh * Tb * d;
    uint32_t* S = Skey + (size_t)warp * Tb;
    const size_t rowoff = (size_t)bh * Tb + row;

    if (active)
        for (int c = lane; c < d; c += 32) qs[warp * d + c] = qb[rowoff * d + c];

    for (int j0 = 0; j0 < Tb; j0 += kSelKeyChunk) {
        const int nk = min(kSelKeyChunk, Tb - j0);
        __syncthreads();
        // float4 loads (d % 4 == 0), unrolled so that each thread's loads are all in flight
        const float4* src4 = reinterpret_cast<const float4*>(kbh + (size_t)j0 * d);
        const int n4 = nk * d / 4;
#pragma unroll 4
        for (int e4 = threadIdx.x; e4 < n4; e4 += kSelWarps * 32) {
            const float4 v = __ldg(src4 + e4);
            const int e = e4 * 4, j = e / d, c = e - j * d;
            kbT[(c + 0) * kLd + j] = v.x;
            kbT[(c + 1) * kLd + j] = v.y;
            kbT[(c + 2) * kLd + j] = v.z;
            kbT[(c + 3) * kLd + j] = v.w;
        }
        __syncthreads();
        if (active) {
            for (int j = lane; j < nk; j += 32) {
                // four interleaved partial sums over d (c = 4t + u), combined in a fixed order
                float a[4] = {0.f, 0.f, 0.f, 0.f};
                int c = 0;
                for (; c + 4 <= d; c += 4)
#pragma unroll
                    for (int u = 0; u < 4; ++u) a[u] = fmaf(qs[warp * d + c + u], kbT[(c + u) * kLd + j], a[u]);
                for (; c < d; ++c) a[0] = fmaf(qs[warp * d + c], kbT[c * kLd + j], a[0]);
                const float acc = (a[0] + a[1]) + (a[2] + a[3]);
                if (scores) scores[rowoff * Tb + j0 + j] = acc;
                S[j0 + j] = sel::order_key(acc);
            }
        }
    }
    __syncwarp();
    if (!active) return;
    int32_t* dst = idx + rowoff * keep;

    if (Tb <= 32) select_rows<1>(S, Tb, keep, lane, dst, 1);
    else if (Tb <= 64) select_rows<2>(S, Tb, keep, lane, dst, 1);
    else if (Tb <= 256) select_rows<8>(S, Tb, keep, lane, dst, 1);
    else {
        // keep-th largest key by MSB-first radix select
        uint32_t prefix = 0, pmask = 0;
        int remaining = keep;
        for (int bit = 31; bit >= 0; --bit) {
            const uint32_t trial = prefix | (1u << bit), tmask = pmask | (1u << bit);
            int c = 0;
            for (int j = lane; j < Tb; j += 32) c += (S[j] & tmask) == trial;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            if (c >= remaining) prefix = trial;
            else remaining -= c;
            pmask = tmask;
        }
        // kept: key > T, or key == T among the first `remaining` equal ones (lowest labels)
        const uint32_t T = prefix;
        int out = 0, eq_seen = 0;
        for (int j0 = 0; j0 < Tb; j0 += 32) {
            const int j = j0 + lane;
            const uint32_t key = j < Tb ? S[j] : 0u;
            const bool gt = j < Tb && key > T;
            const bool eq = j < Tb && key == T;
            const uint32_t eqm = __ballot_sync(0xffffffffu, eq);
            const int eq_rank = eq_seen + __popc(eqm & ((1u << lane) - 1u));
            const bool kept = gt || (eq && eq_rank < remaining);
            const uint32_t km = __ballot_sync(0xffffffffu, kept);
            if (kept) dst[out + __popc(km & ((1u << lane) - 1u))] = j;
            out += __popc(km);
            eq_seen += __popc(eqm);
        }
    }
    if (lane == 0) cnt[rowoff] = keep;
}


constexpr int kFuseCluster = 8;    // CTAs per (batch, head)
// Longest rows of the fused build. With 256 blocks a head (2048 px) its 192 CTAs are 32 rows each and
// fall unevenly on the SMs: 43 us, against 13 (pooling) + 25 (selection) for the two kernels; at 144
// blocks 24 against 21, at 128 22.8 against 25.6; at 64 it takes 8.8 against 4.2 + 6.2. Where its CTAs are
// more than two an SM, rows of more than 64 blocks go to the two kernels as well (mask and forward of
// two images, 81 blocks a head 118.9 -> 114.3 us, 120 blocks 210 -> 202; four images of 64 blocks 182.4
// either way).
constexpr int kFuseMaxTb = 128;

// Affinity row of one query block with the keys held in registers (lane l: labels l + 32 m), then
// the gating. kbs: the head's k_b by rows, the 16-byte chunk c4 of row j at chunk c4 ^ (j & 15) (the 32
// lanes reading one chunk of 32 rows cover all 32 banks: four wavefronts, the least for 512 bytes).
template <int kPer>
__device__ __forceinline__ void affinity_select(const float* q, const float* kbs, int Tb, int keep, int lane,
                                                float* srow, int32_t* dst)
{
    constexpr int kD = 64;
    uint32_t key[kPer];
#pragma unroll
    for (int m = 0; m < kPer; ++m) {
        const int j = lane + 32 * m;
        key[m] = 0u;
        if (j < Tb) {
            const float* row = kbs + j * kD;
            float acc[1];
            sel::affinity<1>(acc, q, kD, [&](int c) {
                return *reinterpret_cast<const float4*>(row + 4 * (c ^ (j & 15)));
            });
            if (srow) srow[j] = acc[0];
            key[m] = sel::order_key(acc[0]);
        }
    }
    sel::ballot_select<kPer>(key, Tb, keep, lane, dst);
}

// One cluster of kFuseCluster CTAs per (batch*head); CTA r of the cluster owns the blocks
// [r * bpc, (r + 1) * bpc) ∩ [0, Tb).
// smem: qown [bpc][64] | kbs [Tb][64] (the head's k_b, 16-byte chunks swizzled by row)
//   1. pool: warp w takes (block, tensor) units w, w + kFuseWarps, ... of its CTA; lane l covers
//      16-byte chunk l % CPR of rows l / CPR + RPI * i, summed in row order, then across
//      lanes by shuffles (fixed order); a q_b mean goes to qown, a k_b mean into kbs of every
//      CTA of the cluster (distributed shared memory stores, one per CTA and chunk).
//   2. one cluster barrier (release / acquire: every CTA's stores into kbs are visible after
//      it, and none follow it, so a CTA may leave once it is done).
//   3. one warp per owned query block: S row by four interleaved partial sums over d, its
//      keys in registers, then the radix walk (affinity_select).
template <typename T, int kFuseWarps, int kMinCtas>
__global__ void __launch_bounds__(kFuseWarps * 32, kMinCtas) ssba_mask_fused_kernel(const T* __restrict__ Q,
                                                                          const T* __restrict__ K, Grid g,
                                                                          int keep, int bpc,
                                                                          int32_t* __restrict__ idx,
                                                                          int32_t* __restrict__ cnt,
                                                                          float* __restrict__ scores)
{
    namespace cg = cooperative_groups;
    constexpr int kD = 64;
    constexpr int VE = Vec<T>::kElems;
    constexpr int CPR = kD / VE;      // 16-byte chunks per token row
    constexpr int RPI = 32 / CPR;     // rows per warp instruction
    constexpr int LOADS = 64 / RPI;   // loads per lane per (block, tensor)
    constexpr int BATCH = LOADS < 16 ? LOADS : 16;  // loads in flight per lane
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ float smf[];
    const int Tb = g.Tb();
    const int rank = (int)cluster.block_rank();
    const int bh = blockIdx.y;
    const int b0 = rank * bpc;
    const int nb = max(0, min(bpc, Tb - b0));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int N = g.H * g.W;
    float* qown = smf;
    float* kbs = qown + bpc * kD;

    // the k_b stores go into the other CTAs' shared memory, which is only valid once every CTA
    // of the cluster runs: arrive here, wait before the first store (after the first loads)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    bool started = false;

    // Q and K may come from the grid launched just before this one
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();

    // 1. pool the owned blocks
    const int col = lane % CPR, r0 = lane / CPR;
    for (int u = warp; u < 2 * nb; u += kFuseWarps) {
        const int which = u & 1, k = u >> 1, label = b0 + k;
        const T* X = (which ? K : Q) + (size_t)bh * N * kD + col * VE;
        // window origin in the rolled frame, once per unit; rows and columns of the 8x8
        // window then follow by shifts (the same map as Grid::token with blk = 8)
        const int br = label / g.bw, bc = label - br * g.bw;
        const int rb = br * 8 - g.sr, cb = bc * 8 - g.sc;
        float acc[VE];
#pragma unroll
        for (int e = 0; e < VE; ++e) acc[e] = 0.f;
#pragma unroll
        for (int i0 = 0; i0 < LOADS; i0 += BATCH) {
            uint4 v[BATCH];
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int pos = r0 + (i0 + i) * RPI;
                int r = rb + (pos >> 3), c = cb + (pos & 7);
                r += r < 0 ? g.H : 0;
                c += c < 0 ? g.W : 0;
                v[i] = __ldg(reinterpret_cast<const uint4*>(X + (size_t)(r * g.W + c) * kD));
            }
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                float f[VE];
                Vec<T>::to_f32(v[i], f);
#pragma unroll
                for (int e = 0; e < VE; ++e) acc[e] += f[e];
            }
        }
#pragma unroll
        for (int o = CPR; o < 32; o <<= 1)
#pragma unroll
            for (int e = 0; e < VE; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
        if (!started) {  // warp-uniform
            asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
            started = true;
        }
        if (r0 == 0) {
#pragma unroll
            for (int e = 0; e < VE; ++e) acc[e] *= 1.0f / 64.0f;
            if (!which) {
                float* dst = qown + k * kD + col * VE;
#pragma unroll
                for (int e = 0; e < VE; ++e) dst[e] = acc[e];
            } else {
                // chunks col * VE / 4 .. of row `label`, into the k_b of every CTA of the cluster
#pragma unroll
                for (int r = 0; r < kFuseCluster; ++r) {
                    float* rk = cluster.map_shared_rank(kbs, r) + label * kD;
#pragma unroll
                    for (int h = 0; h < VE / 4; ++h) {
                        const int c4 = col * (VE / 4) + h;
                        *reinterpret_cast<float4*>(rk + 4 * (c4 ^ (label & 15))) =
                            make_float4(acc[4 * h], acc[4 * h + 1], acc[4 * h + 2], acc[4 * h + 3]);
                    }
                }
            }
        }
    }
    if (!started) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    // 2. every k_b row of the head is in this CTA's kbs after the barrier
    cluster.sync();

    // 3. affinity rows and selection
    for (int k = warp; k < nb; k += kFuseWarps) {
        const size_t rowoff = (size_t)bh * Tb + b0 + k;
        const float* q = qown + k * kD;
        float* srow = scores ? scores + rowoff * Tb : nullptr;
        int32_t* dst = idx + rowoff * keep;
        if (Tb <= 32) affinity_select<1>(q, kbs, Tb, keep, lane, srow, dst);
        else if (Tb <= 64) affinity_select<2>(q, kbs, Tb, keep, lane, srow, dst);
        else affinity_select<4>(q, kbs, Tb, keep, lane, srow, dst);
        if (lane == 0) cnt[rowoff] = keep;
    }
}

// Block means alone, with the pooling loop of ssba_mask_fused_kernel (so the same inputs give
// bit-identical means): CTA = kPoolWin blocks of one (batch*head), warp w pools tensor (w & 1)
// of block w / 2, every load of a lane in flight at once; programmatic dependent launch.
constexpr int kPoolWin = 4;
template <typename T>
__global__ void __launch_bounds__(2 * kPoolWin * 32) ssba_pool_blocks_kernel(const T* __restrict__ Q,
                                                                             const T* __restrict__ K, Grid g,
                                                                             float* __restrict__ qb,
                                                                             float* __restrict__ kb)
{
    constexpr int kD = 64;
    constexpr int VE = Vec<T>::kElems;
    constexpr int CPR = kD / VE;
    constexpr int RPI = 32 / CPR;
    constexpr int LOADS = 64 / RPI;
    constexpr int BATCH = LOADS < 16 ? LOADS : 16;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int Tb = g.Tb();
    const int label = blockIdx.x * kPoolWin + (warp >> 1), which = warp & 1, bh = blockIdx.y;
    const int N = g.H * g.W;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (label >= Tb) return;
    const int col = lane % CPR, r0 = lane / CPR;
    const T* X = (which ? K : Q) + (size_t)bh * N * kD + col * VE;
    const int br = label / g.bw, bc = label - br * g.bw;
    const int rb = br * 8 - g.sr, cb = bc * 8 - g.sc;
    float acc[VE];
#pragma unroll
    for (int e = 0; e < VE; ++e) acc[e] = 0.f;
#pragma unroll
    for (int i0 = 0; i0 < LOADS; i0 += BATCH) {
        uint4 v[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            const int pos = r0 + (i0 + i) * RPI;
            int r = rb + (pos >> 3), c = cb + (pos & 7);
            r += r < 0 ? g.H : 0;
            c += c < 0 ? g.W : 0;
            v[i] = __ldg(reinterpret_cast<const uint4*>(X + (size_t)(r * g.W + c) * kD));
        }
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            float f[VE];
            Vec<T>::to_f32(v[i], f);
#pragma unroll
            for (int e = 0; e < VE; ++e) acc[e] += f[e];
        }
    }
#pragma unroll
    for (int o = CPR; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < VE; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    if (r0 == 0) {
        float* dst = (which ? kb : qb) + ((size_t)bh * Tb + label) * kD + col * VE;
#pragma unroll
        for (int e = 0; e < VE; ++e) dst[e] = acc[e] * (1.0f / 64.0f);
    }
}

}  // namespace

int launch_pool_blocks(const ssba_desc& d, const Grid& g, const void* Q, const void* K, float* qb, float* kb,
                       cudaStream_t st)
{
    if (d.head_dim != 64 || g.blk != 8) return launch_pool(d, g, Q, K, qb, kb, st);
    const int BH = d.B * d.heads;
    const size_t head = (size_t)g.H * g.W * 64, means = (size_t)g.Tb() * 64;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(2 * kPoolWin * 32, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    for (int h0 = 0; h0 < BH; h0 += kMaxGridY) {
        cfg.gridDim = dim3((g.Tb() + kPoolWin - 1) / kPoolWin, min(kMaxGridY, BH - h0), 1);
        auto launch = [&](auto kernel, auto* x) {
            return cudaLaunchKernelEx(&cfg, kernel, x + h0 * head, static_cast<decltype(x)>(K) + h0 * head, g,
                                      qb + h0 * means, kb + h0 * means);
        };
        cudaError_t e = d.dtype == SSBA_BF16
                            ? launch(ssba_pool_blocks_kernel<__nv_bfloat16>, static_cast<const __nv_bfloat16*>(Q))
                            : launch(ssba_pool_blocks_kernel<float>, static_cast<const float*>(Q));
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) {
            set_error("ssba_pool_blocks_kernel launch: %s", cudaGetErrorString(e));
            return SSBA_ERR_CUDA;
        }
    }
    return SSBA_OK;
}

int launch_pool(const ssba_desc& d, const Grid& g, const void* Q, const void* K, float* qb, float* kb,
                cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    if (d.head_dim == 64 && g.blk == 8) {
        dim3 grid(g.Tb(), d.B * d.heads);
        if (d.dtype == SSBA_BF16)
            ssba_pool_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(Q),
                                                                  static_cast<const __nv_bfloat16*>(K), g, qb, kb);
        else
            ssba_pool_kernel<float><<<grid, 256, 0, st>>>(static_cast<const float*>(Q), static_cast<const float*>(K),
                                                          g, qb, kb);
        e = cudaGetLastError();
    } else {
        const int P = g.blk * g.blk;
        const size_t smem = (size_t)2 * P * d.head_dim * sizeof(float);
        if (smem > kPoolSmem) {
            set_error("ssba_build_mask: block*block*head_dim too large for the pooling kernel");
            return SSBA_ERR_UNSUPPORTED;
        }
        static PerDeviceOnce attr;
        attr.run([] {
            const int n = (int)kPoolSmem;
            cudaFuncSetAttribute(ssba_pool_generic_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
            cudaFuncSetAttribute(ssba_pool_generic_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
        });
        dim3 grid(g.Tb(), d.B * d.heads);
        if (d.dtype == SSBA_BF16) {
            auto k = ssba_pool_generic_kernel<__nv_bfloat16>;
            k<<<grid, 128, smem, st>>>(static_cast<const __nv_bfloat16*>(Q), static_cast<const __nv_bfloat16*>(K), g,
                                       d.head_dim, qb, kb);
        } else {
            auto k = ssba_pool_generic_kernel<float>;
            k<<<grid, 128, smem, st>>>(static_cast<const float*>(Q), static_cast<const float*>(K), g, d.head_dim, qb,
                                       kb);
        }
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error("ssba_pool_kernel launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

int launch_select(const ssba_desc& d, const Grid& g, int keep, const float* qb, const float* kb,
                  int32_t* idx, int32_t* cnt, float* scores, cudaStream_t st)
{
    const int Tb = g.Tb();
    if (Tb > kMaxTb) {
        set_error("ssba_build_mask: Tb=%d exceeds the selection kernel's limit of %d blocks", Tb, kMaxTb);
        return SSBA_ERR_UNSUPPORTED;
    }
    if (d.head_dim == 64) {
        const int BH = d.B * d.heads;
        // Rows a warp. Short rows: two where a CTA's eight warps of one each would be many CTAs an SM (24 heads,
        // us, one row and two: 64 blocks 4.9, 5.1; at batch 4 9.9, 9.1; 256 blocks 25, 20), one below and up to 32
        // blocks, where a row is little work (16 blocks at batch 8 5.4, 5.6). Rows of 257 to 1024: the fewest
        // that leave a CTA an SM, since a warp's rows follow each other (one head of 510 blocks 15, 19
        // and 25 us for one, two and four; 24 heads 78, 61, 54). Longer ones: two, what their keys leave room for
        // (1280 blocks, 24 heads 726, 483; one head 55, 50).
        const int sms = device_sm_count();
        auto ctas = [&](int r) { return (long long)BH * ((Tb + kSelWarps * r - 1) / (kSelWarps * r)); };
        const int rows = Tb <= 32     ? 1
                         : Tb <= 256  ? ((long long)BH * Tb >= 10ll * sms ? 2 : 1)
                         : Tb <= 1024 ? (ctas(1) <= sms ? 1 : (ctas(2) <= sms ? 2 : 4))
                                      : 2;
        const int per = Tb <= 32 ? 1 : (Tb <= 256 ? 8 : (Tb <= 512 ? 16 : (Tb <= 1024 ? 32 : 64)));
        struct Variant {
            int rows, per, longest;  // longest row it is given
            decltype(&ssba_select64_kernel<1, 1>) kernel;
        };
        static const Variant variants[] = {
            {1, 1, 32, ssba_select64_kernel<1, 1>},     {1, 8, 256, ssba_select64_kernel<1, 8>},
            {2, 8, 256, ssba_select64_kernel<2, 8>},    {1, 16, 512, ssba_select64_kernel<1, 16>},
            {2, 16, 512, ssba_select64_kernel<2, 16>},  {4, 16, 512, ssba_select64_kernel<4, 16>},
            {1, 32, 1024, ssba_select64_kernel<1, 32>}, {2, 32, 1024, ssba_select64_kernel<2, 32>},
            {4, 32, 1024, ssba_select64_kernel<4, 32>}, {2, 64, kMaxTb, ssba_select64_kernel<2, 64>},
        };
        // the largest size of each, once: a limit set for each call could be lowered by another thread before
        // this one's launch
        static PerDeviceOnce attr64;
        attr64.run([] {
            for (const Variant& v : variants)
                cudaFuncSetAttribute(v.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sel64_smem(v.rows, v.longest));
        });
        const Variant* v = variants;
        while (v->rows != rows || v->per != per) ++v;
        const int cta = kSelWarps * rows;
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(kSelWarps * 32, 1, 1);
        cfg.dynamicSmemBytes = sel64_smem(rows, Tb);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        for (int h0 = 0; h0 < BH; h0 += kMaxGridY) {
            const size_t row = (size_t)h0 * Tb;
            cfg.gridDim = dim3((Tb + cta - 1) / cta, min(kMaxGridY, BH - h0), 1);
            cudaError_t e = cudaLaunchKernelEx(&cfg, v->kernel, qb + row * 64, kb + row * 64, Tb, keep, idx + row * keep,
                                               cnt + row, scores ? scores + row * Tb : nullptr);
            if (e == cudaSuccess) e = cudaGetLastError();
            if (e != cudaSuccess) {
                set_error("ssba_select64_kernel launch: %s", cudaGetErrorString(e));
                return SSBA_ERR_CUDA;
            }
        }
        return SSBA_OK;
    }
    size_t smem = ((size_t)d.head_dim * (kSelKeyChunk + 1) + (size_t)kSelWarps * d.head_dim +
                   (size_t)kSelWarps * Tb) * sizeof(float);
    if (smem > kSelSmem) {
        set_error("ssba_build_mask: selection working set too large (%zu bytes)", smem);
        return SSBA_ERR_UNSUPPORTED;
    }
    static PerDeviceOnce attr;
    attr.run([] {
        cudaFuncSetAttribute(ssba_select_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
        cudaFuncSetAttribute(ssba_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSelSmem);
    });
    dim3 grid((Tb + kSelWarps - 1) / kSelWarps, d.B * d.heads);
    ssba_select_kernel<<<grid, kSelWarps * 32, smem, st>>>(qb, kb, Tb, d.head_dim, keep, idx, cnt, scores);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("ssba_select_kernel launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

}  // namespace ssba

namespace ssba {

// The fused mask build (one launch) when the shape allows it; returns SSBA_ERR_UNSUPPORTED
// (without launching and without setting an error) otherwise.
int launch_mask_fused(const ssba_desc& d, const Grid& g, int keep, const void* Q, const void* K, int32_t* idx,
                      int32_t* cnt, float* scores, cudaStream_t st)
{
    const int Tb = g.Tb();
    const bool spread = d.B * d.heads * kFuseCluster <= 2 * device_sm_count();
    if (d.head_dim != 64 || g.blk != 8 || Tb > (spread ? kFuseMaxTb : 64)) return SSBA_ERR_UNSUPPORTED;
    const int bpc = (Tb + kFuseCluster - 1) / kFuseCluster;
    const size_t smem = ((size_t)bpc * 64 + (size_t)Tb * 64) * sizeof(float);
    static_assert((kFuseMaxTb / kFuseCluster + kFuseMaxTb) * 64 * sizeof(float) <= 48 * 1024, "no opt-in needed");
    // CTAs an SM. A grid of up to two an SM takes the instantiation whose 128 registers (kMinCtas 2) let two and
    // no more share one, so that its clusters spread; left to itself the compiler takes 80, three fit,
    // and clusters crowd some SMs while others idle. Two against three, 24 heads, GPU time: 1024 px mask and
    // forward 44.2 against 47.1 us, the mask alone 8.4 either way (28 heads 8.5 against 10.5); 99 blocks 80
    // against 87 together. (Asking for 80 KB of shared memory spreads them too, but with 80 registers fewer
    // loads are in flight: alone 8.8 us, fp32 9.5 against 8.7, 36 heads 11.5 against 8.9.) Grids above two
    // an SM have more than one round of two and are faster with three (four 1024 px images 29.9 -> 28.7).
    // Warps of a CTA: one per block, where a CTA's nine to twelve blocks would be two rounds of eight warps
    // (768 x 1408 px, 66 blocks, mask and forward 54.5 -> 52.0 us, 1152 px 67.6 -> 65.9; 16 warps 54.5 and
    // 68.1). At up to eight blocks the four more are idle and only cost room (512 px 14.8 either way, four
    // 1024 px images 183 -> 188).
    const bool wide = bpc > 8 && bpc <= 12;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kFuseCluster, d.B * d.heads, 1);
    cfg.blockDim = dim3(wide ? 12 * 32 : 8 * 32, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kFuseCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see grid_dep_wait
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    auto launch = [&](auto kernel, auto q, auto k) {
        return cudaLaunchKernelEx(&cfg, kernel, q, k, g, keep, bpc, idx, cnt, scores);
    };
    const cudaError_t e =
        d.dtype == SSBA_BF16
            ? launch(wide     ? ssba_mask_fused_kernel<__nv_bfloat16, 12, 0>
                     : spread ? ssba_mask_fused_kernel<__nv_bfloat16, 8, 2>
                              : ssba_mask_fused_kernel<__nv_bfloat16, 8, 0>,
                     static_cast<const __nv_bfloat16*>(Q), static_cast<const __nv_bfloat16*>(K))
            : launch(wide     ? ssba_mask_fused_kernel<float, 12, 0>
                     : spread ? ssba_mask_fused_kernel<float, 8, 2>
                              : ssba_mask_fused_kernel<float, 8, 0>,
                     static_cast<const float*>(Q), static_cast<const float*>(K));
    if (e != cudaSuccess) {
        set_error("ssba_mask_fused_kernel launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

}  // namespace ssba
