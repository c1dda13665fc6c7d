// attn_dense.cu -- dense bf16 softmax attention on the sm_103a tensor cores: the 0 % sparsity
// baseline of Table 2 (every key of the head), the denominator of the sparse kernel's speed-up.
//
// Without index lists every query shares every key, so tiles are 128 contiguous tokens:
//   S = Q_u K_j^T   tcgen05.mma kind::f16, M=128 N=128 K=16 x 4 (A = Q tile, B = K tile, both
//                   K-major SW128 in shared memory)
//   O += P V_j      M=128 N=64 K=16 x 8 (A = P, bf16, from tensor memory; B = V tile MN-major)
// Work unit = one tile of 128 query rows of one (batch, head); it visits all N/128 key tiles.
// Persistent CTAs, one per SM (their shared memory fills it), each running two independent
// streams of units (unit v + r V for stream v of V), warp-specialised, 8 warps a stream (512
// threads, 128 registers each):
//   K producer, V producer   TMA: the unit's Q tile, then the key tiles into rings of three 16 KB
//                  stages each (128-row boxes of a [B*heads][N][64] map)
//   QK issuer      QK_j once the softmax has read S_{j-1}
//   PV issuer      PV_j once P_j is stored and V_j has landed
//   softmax        four warps, one thread per row (TMEM lane). Exp2 in the log2-scaled domain against a
//                  reference max m, the first tile's row maximum: a tile's 128 scores are read once, in
//                  four 32-column chunks, and become P at once. S is released when the last chunk is
//                  in registers and the first three have been seen to sum to at most 2^24; where they
//                  do not, the tile's maximum is taken, m raised, O rescaled and P formed again (as in
//                  attn_tc.cu); where the last chunk alone does not, m is raised by a whole number and
//                  P rescaled. At the end of a unit they write O / l in bf16 and lse.
// TMEM of a stream: S 128 + P 64 (bf16 pairs) + O 64 = 256 columns; the two streams take 512.
// What bounds it: a tile takes about 1050 cycles of an SM, of which the tensor pipe is busy 608 (QK 4 x
// 80, PV 8 x 36) and a scheduler's softmax warps about 800 (128 exp2s a row and what is around them).
// 24 heads: 1024 px 137 -> 98 us (1050 TFLOP/s; its last round of tiles leaves half the SMs idle), 2048
// px 1852 -> 1310 us (1260 TFLOP/s), against the kernel that read S twice (maximum, then exp2s), had
// one issuer for both products and 2-stage rings. With the wait for P's buffer in front of a tile's
// exp2s instead of its second chunk's store: 115 and 1500. (In front of the first chunk's store: 101 and
// 1330; of the third's: as of the second's.) Releasing S only after the last exp2s: 131 and 1772;
// already when half of it is formed and the rest in registers: 2 % slower than as it is.
// Every wait is bounded (globaltimer budget + CTA abort flag); a timeout is reported in
// the device status word and the roles drain their copies and products before the CTA exits.
#include <cuda.h>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "ptx.cuh"

namespace ssba {
namespace {

using namespace ptx;

constexpr int kD = 64;
constexpr int kTile = 128;                        // query rows of a unit = keys of a key tile
constexpr uint32_t kTileBytes = kTile * kD * 2;   // 16 KB
constexpr int kStages = 3;                        // K and V rings
constexpr int kStreams = 2;
constexpr int kSoftWarps = 4;                     // softmax warps of a stream
constexpr int kRoleWarps = 4;                     // K producer, QK issuer, V producer, PV issuer of a stream
constexpr int kThreads = kStreams * (kSoftWarps + kRoleWarps) * 32;
enum Role { kLoadK = 0, kQK = 1, kLoadV = 2, kPV = 3, kSoftmax = 4 };
constexpr uint32_t kStreamCols = 256;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0;    // [0,128)
constexpr uint32_t kColP = 128;  // [128,192)
constexpr uint32_t kColO = 192;  // [192,256)
constexpr float kRaise = 16777216.f;  // 2^24: row sum of a tile above which the reference max is raised
constexpr uint32_t kIdescQK = idesc_bf16_f32(128, 128, false, false);
constexpr uint32_t kIdescPV = idesc_bf16_f32(128, 64, false, true);

struct __align__(1024) StreamSmem {
    uint8_t q[kTileBytes];
    uint8_t k[kStages][kTileBytes];
    uint8_t v[kStages][kTileBytes];
};

struct StreamCtl {
    uint64_t q_full, q_empty;
    uint64_t k_full[kStages], k_empty[kStages];
    uint64_t v_full[kStages], v_empty[kStages];
    uint64_t s_full;  // QK_g has finished
    uint64_t s_free;  // the four softmax warps have read S_g
    uint64_t p_full;  // the four softmax warps have stored P_g (and read the last unit's O)
    uint64_t o_full;  // PV_g has finished
    uint64_t drain[2];
};

struct __align__(1024) DenseSmem {
    StreamSmem st[kStreams];
    StreamCtl ctl[kStreams];
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(DenseSmem) + 1024 <= 232448, "shared memory of one CTA (227 KB opt-in limit)");

struct DenseParams {
    __nv_bfloat16* O;
    float* lse;
    int BH;           // batch * heads
    int N;            // tokens, a multiple of 128
    int nt;           // N / 128 tiles a head
    int units;        // BH * nt
    float scale_log2; // softmax scale * log2(e)
    int* status;
    uint64_t budget_ns;
};

struct DenseMaps {
    CUtensorMap q, k, v;
};

__device__ __forceinline__ float fast_exp2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ bool wait_raw(uint32_t bar, uint32_t parity, uint64_t budget_ns)
{
    const uint64_t t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity))
        if (globaltimer_ns() - t0 > budget_ns) return false;
    return true;
}

// Units of stream v (V streams): v, v + V, v + 2V, ...
__device__ __forceinline__ int stream_units(const DenseParams& p, int v, int V)
{
    return p.units > v ? (p.units - v + V - 1) / V : 0;
}

__global__ void __launch_bounds__(kThreads, 1) ssba_dense_tc_kernel(const __grid_constant__ DenseMaps maps,
                                                                    const DenseParams p)
{
    extern __shared__ uint8_t smem_raw[];
    DenseSmem& cs = *reinterpret_cast<DenseSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                  ~static_cast<uintptr_t>(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        cs.abort_flag = 0;
        for (int s = 0; s < kStreams; ++s) {
            StreamCtl& c = cs.ctl[s];
            for (int b = 0; b < kStages; ++b) {
                mbar_init(smem_u32(&c.k_full[b]), 1);
                mbar_init(smem_u32(&c.k_empty[b]), 1);
                mbar_init(smem_u32(&c.v_full[b]), 1);
                mbar_init(smem_u32(&c.v_empty[b]), 1);
            }
            mbar_init(smem_u32(&c.q_full), 1);
            mbar_init(smem_u32(&c.q_empty), 1);
            mbar_init(smem_u32(&c.s_full), 1);
            mbar_init(smem_u32(&c.s_free), kSoftWarps);
            mbar_init(smem_u32(&c.p_full), kSoftWarps);
            mbar_init(smem_u32(&c.o_full), 1);
            mbar_init(smem_u32(&c.drain[0]), 1);
            mbar_init(smem_u32(&c.drain[1]), 1);
        }
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&cs.tmem_base), kTmemCols);
        tmem_relinquish();
    }
    if (warp == 2 && lane == 0) {
        tma_prefetch_desc(&maps.q);
        tma_prefetch_desc(&maps.k);
        tma_prefetch_desc(&maps.v);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // everything above reads no input (programmatic dependent launch: inputs may come from the
    // grid launched before this one)
    grid_dep_wait();
    grid_dep_launch();
    // the softmax warps first, so that a stream's four are one per TMEM lane quadrant
    const bool soft = warp < kStreams * kSoftWarps;
    const int stream = soft ? warp / kSoftWarps : (warp - kStreams * kSoftWarps) / kRoleWarps;
    const int role = soft ? kSoftmax : (warp - kStreams * kSoftWarps) % kRoleWarps;
    StreamSmem& sm = cs.st[stream];
    StreamCtl& ct = cs.ctl[stream];
    const int V = gridDim.x * kStreams;
    const int v = stream * gridDim.x + blockIdx.x;  // stream-major numbering of the grid's streams
    const int nunits = stream_units(p, v, V);
    const uint32_t tbase = cs.tmem_base + stream * kStreamCols;
    volatile int* abortf = &cs.abort_flag;
    const uint32_t abort_at = smem_u32(&cs.abort_flag);
    bool dead = false;
    uint32_t g = 0;  // key tiles that the role is through with
    int nq = 0;      // (K producer) units whose Q is announced

    if (role == kLoadK || role == kLoadV) {
        // ------------------------------------------------------------ TMA producers
        const bool is_k = role == kLoadK;
        const uint32_t empty0 = smem_u32(is_k ? &ct.k_empty[0] : &ct.v_empty[0]);
        const uint32_t full0 = smem_u32(is_k ? &ct.k_full[0] : &ct.v_full[0]);
        const uint32_t tile0 = smem_u32(is_k ? &sm.k[0][0] : &sm.v[0][0]);
        const CUtensorMap* map = is_k ? &maps.k : &maps.v;
        if (lane == 0) {
            for (int n = 0; n < nunits && !dead; ++n) {
                const int u = v + n * V, bh = u / p.nt, qt = u - bh * p.nt;
                for (int j = 0; j < p.nt; ++j) {
                    const uint32_t st = g % kStages;
                    if (!mbar_wait(empty0 + 8 * st, ((g / kStages) & 1) ^ 1, abortf, p.budget_ns)) {
                        dead = true;
                        break;
                    }
                    mbar_arrive_expect_tx(full0 + 8 * st, kTileBytes);
                    tma_load_3d(tile0 + st * kTileBytes, map, full0 + 8 * st, 0, j * kTile, bh);
                    ++g;
                    if (is_k && j == 0) {  // the unit's Q after its first K: it waits longest
                        if (!mbar_wait(smem_u32(&ct.q_empty), (n & 1) ^ 1, abortf, p.budget_ns)) {
                            dead = true;
                            break;
                        }
                        mbar_arrive_expect_tx(smem_u32(&ct.q_full), kTileBytes);
                        tma_load_3d(smem_u32(&sm.q[0]), &maps.q, smem_u32(&ct.q_full), 0, qt * kTile, bh);
                        ++nq;
                    }
                }
            }
        }
        __syncwarp();
    } else if (role == kQK) {
        // ------------------------------------------------------------ QK issuer
        for (int n = 0; n < nunits && !*abortf; ++n) {
            wait_phase(smem_u32(&ct.q_full), n & 1, abort_at, p.budget_ns);
            for (int j = 0; j < p.nt; ++j, ++g) {
                const uint32_t st = g % kStages;
                wait_phase(smem_u32(&ct.k_full[st]), (g / kStages) & 1, abort_at, p.budget_ns);
                if (g >= 1) wait_phase(smem_u32(&ct.s_free), (g - 1) & 1, abort_at, p.budget_ns);
                tc_fence_after();
                if (elect_one_sync()) {
                    const uint64_t adesc = sdesc_sw128(smem_u32(&sm.q[0]), 16, 1024);
                    const uint64_t bdesc = sdesc_sw128(smem_u32(&sm.k[st][0]), 16, 1024);
#pragma unroll
                    for (int k = 0; k < kD / 16; ++k)
                        mma_ss(tbase + kColS, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), kIdescQK,
                               k > 0 ? 1u : 0u);
                    mma_commit(smem_u32(&ct.s_full));
                    mma_commit(smem_u32(&ct.k_empty[st]));
                    if (j == p.nt - 1) mma_commit(smem_u32(&ct.q_empty));
                }
                __syncwarp();
            }
        }
        dead = *abortf != 0;
    } else if (role == kPV) {
        // ------------------------------------------------------------ PV issuer
        for (int n = 0; n < nunits && !*abortf; ++n)
            for (int j = 0; j < p.nt; ++j, ++g) {
                const uint32_t st = g % kStages;
                wait_phase(smem_u32(&ct.v_full[st]), (g / kStages) & 1, abort_at, p.budget_ns);
                wait_phase(smem_u32(&ct.p_full), g & 1, abort_at, p.budget_ns);
                tc_fence_after();
                if (elect_one_sync()) {
                    const uint64_t vdesc = sdesc_sw128(smem_u32(&sm.v[st][0]), 8192, 1024);
#pragma unroll
                    for (int k = 0; k < kTile / 16; ++k)
                        mma_ts(tbase + kColO, tbase + kColP + k * 8, vdesc + (uint64_t)(k * 128), kIdescPV,
                               (j > 0 || k > 0) ? 1u : 0u);
                    mma_commit(smem_u32(&ct.o_full));
                    mma_commit(smem_u32(&ct.v_empty[st]));
                }
                __syncwarp();
            }
        dead = *abortf != 0;
    } else {
        // ------------------------------------------------------------ softmax and output
        const int quad = warp & 3, row = quad * 32 + lane;
        const uint32_t tq = tbase + (static_cast<uint32_t>(quad * 32) << 16);
        const uint32_t scol = tq + kColS, pcol = tq + kColP, ocol = tq + kColO;
        const float c = p.scale_log2;
        for (int n = 0; n < nunits && !*abortf; ++n) {
            float m_used = 0.f, l = 0.f;
            for (int j = 0; j < p.nt; ++j, ++g) {
                wait_phase(smem_u32(&ct.s_full), g & 1, abort_at, p.budget_ns);
                tc_fence_after();
                const float2 c2 = make_float2(c, c);
                // P = exp2(s c - m) of one chunk in bf16 to tensor memory, its row sum onto ls2
                float2 ls2[2];
                uint32_t pk0[16];  // chunk 0 of P, until the buffer is free
                auto exps = [&](int ch, const uint32_t (&r)[32]) {
                    const float2 nm2 = make_float2(-m_used, -m_used);
                    uint32_t pk[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float2 x = __ffma2_rn(
                            make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])), c2, nm2);
                        const float2 pp = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                        ls2[e & 1] = __fadd2_rn(ls2[e & 1], pp);
                        pk[e] = pack_bf16(pp.x, pp.y);
                    }
                    if (ch == 0) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) pk0[e] = pk[e];
                        return;
                    }
                    // P's buffer is free once PV_{g-1} has finished (O then holds every earlier PV)
                    if (ch == 1) {
                        if (g >= 1) wait_phase(smem_u32(&ct.o_full), (g - 1) & 1, abort_at, p.budget_ns);
                        tc_fence_after();
                        tmem_st_32x32b_x16(pcol, pk0);
                    }
                    tmem_st_32x32b_x16(pcol + 16 * ch, pk);
                };
                auto sum = [&] { return (ls2[0].x + ls2[1].x) + (ls2[0].y + ls2[1].y); };
                auto rescale_o = [&](float alpha) {  // PV_{g-1} has finished
#pragma unroll
                    for (int h2 = 0; h2 < 4; ++h2) {
                        uint32_t o[16];
                        tmem_ld_32x32b_x16(ocol + h2 * 16, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st_32x32b_x16(ocol + h2 * 16, o);
                    }
                };
                uint32_t r[32];
                // chunks 0-2; the first tile takes its maximum first, and so does a tile whose sum
                // comes out too large (S is still there)
                bool over = j == 0;
#pragma unroll 1
                for (bool raise = j == 0;; raise = true) {
                    if (raise) {
                        float mx = -INFINITY;
#pragma unroll
                        for (int ch = 0; ch < 4; ++ch) {
                            tmem_ld_32x32b_x32(scol + 32 * ch, r);
                            tmem_wait_ld();
                            float t4[4] = {mx, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                            for (int e = 0; e < 32; e += 2)
                                t4[(e >> 1) & 3] = max3(t4[(e >> 1) & 3], __uint_as_float(r[e]), __uint_as_float(r[e + 1]));
                            mx = fmaxf(fmaxf(t4[0], t4[1]), fmaxf(t4[2], t4[3]));
                        }
                        const float mx2 = fmaxf(mx * c, -3.0e38f);  // finite, so that scores of -inf give P = 0
                        const float alpha = over && j > 0 ? fast_exp2(m_used - mx2) : 1.f;
                        m_used = over ? mx2 : m_used;
                        l *= alpha;
                        if (j > 0) {
                            wait_phase(smem_u32(&ct.o_full), (g - 1) & 1, abort_at, p.budget_ns);
                            tc_fence_after();
                            rescale_o(alpha);
                        }
                    }
                    ls2[0] = ls2[1] = make_float2(0.f, 0.f);
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        tmem_ld_32x32b_x32(scol + 32 * ch, r);
                        tmem_wait_ld();
                        exps(ch, r);
                    }
                    tmem_ld_32x32b_x32(scol + 96, r);
                    over = !(sum() <= kRaise);
                    tmem_wait_ld();
                    if (raise || !__any_sync(0xffffffffu, over)) break;
                }
                const float ls012 = sum();
                // S is read in full: QK_{g+1} may overwrite it
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ct.s_free));
                exps(3, r);
                float ls = sum();
                over = j > 0 && !(ls <= kRaise);
                if (__any_sync(0xffffffffu, over)) {
                    // the last chunk alone came out too large: m is raised by a whole number, so that the
                    // rest of P (bf16) is rescaled exactly; or, where nothing of that rest is left (alpha is 0),
                    // to the chunk's maximum itself, as the sum with a very low m (scores of -inf, or of -1e10)
                    // would not hold it
                    float mx = __uint_as_float(r[0]);
#pragma unroll
                    for (int e = 1; e < 32; ++e) mx = fmaxf(mx, __uint_as_float(r[e]));
                    const float up = over ? fmaxf(ceilf(mx * c - m_used), 0.f) : 0.f;
                    const float alpha = fast_exp2(-up);
                    rescale_o(alpha);
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        uint32_t pk[16];
                        tmem_wait_st();
                        tmem_ld_32x32b_x16(pcol + 16 * ch, pk);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            pk[e] = pack_bf16(__uint_as_float(pk[e] << 16) * alpha,
                                              __uint_as_float(pk[e] & 0xffff0000u) * alpha);
                        tmem_st_32x32b_x16(pcol + 16 * ch, pk);
                    }
                    l *= alpha;
                    ls2[0] = ls2[1] = make_float2(0.f, 0.f);
                    m_used = up > 256.f ? mx * c : m_used + up;
                    exps(3, r);
                    ls = sum() + ls012 * alpha;
                }
                l += ls;
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ct.p_full));
            }
            // the unit's rows: O / l in bf16 (two halves of 32 columns) and lse, after its last PV
            const int u = v + n * V, bh = u / p.nt, qt = u - bh * p.nt;
            wait_phase(smem_u32(&ct.o_full), (g - 1) & 1, abort_at, p.budget_ns);
            tc_fence_after();
            const bool ok = l > 0.f;
            const float inv = ok ? 1.f / l : 0.f;
            const size_t tok = (size_t)bh * p.N + (size_t)qt * kTile + row;
            uint4* dst = reinterpret_cast<uint4*>(p.O + tok * kD);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t o[32];
                tmem_ld_32x32b_x32(ocol + 32 * h, o);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint4 w;
                    w.x = pack_bf16(__uint_as_float(o[8 * i + 0]) * inv, __uint_as_float(o[8 * i + 1]) * inv);
                    w.y = pack_bf16(__uint_as_float(o[8 * i + 2]) * inv, __uint_as_float(o[8 * i + 3]) * inv);
                    w.z = pack_bf16(__uint_as_float(o[8 * i + 4]) * inv, __uint_as_float(o[8 * i + 5]) * inv);
                    w.w = pack_bf16(__uint_as_float(o[8 * i + 6]) * inv, __uint_as_float(o[8 * i + 7]) * inv);
                    dst[4 * h + i] = w;
                }
            }
            p.lse[tok] = ok ? (m_used * 0.69314718055994531f + logf(l)) : -INFINITY;
            tc_fence_before();  // the next unit's first PV, which waits for p_full, overwrites O
        }
        dead = *abortf != 0;
    }
    if (__syncthreads_or(dead)) {
        // a wait ran out: nothing more is issued, but a role that was done before may have left copies or products in
        // flight, which the ones that gave up have not waited for
        if ((role == kLoadK || role == kLoadV) && lane == 0) {
            const uint32_t full0 = smem_u32(role == kLoadK ? &ct.k_full[0] : &ct.v_full[0]);
            for (uint32_t x = g > kStages ? g - kStages : 0; x < g; ++x)
                wait_raw(full0 + 8 * (x % kStages), (x / kStages) & 1, p.budget_ns);
            if (nq > 0) wait_raw(smem_u32(&ct.q_full), (nq - 1) & 1, p.budget_ns);
        }
        if ((role == kQK || role == kPV) && elect_one_sync()) {
            const uint32_t bar = smem_u32(&ct.drain[role == kPV]);
            mma_commit(bar);
            wait_raw(bar, 0, p.budget_ns);
        }
        if (threadIdx.x == 0) atomicExch(p.status, SSBA_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(cs.tmem_base, kTmemCols);
}

// [B*heads][N][64] bf16 as a 3-D map with 128-row boxes (128-byte swizzle).
bool encode_tile_map(CUtensorMap* m, const void* base, int BH, int N)
{
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)kD, (cuuint64_t)N, (cuuint64_t)BH};
    cuuint64_t strides[2] = {(cuuint64_t)kD * 2, (cuuint64_t)N * kD * 2};
    cuuint32_t box[3] = {kD, kTile, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

PerDeviceOnce g_dense_attr;

}  // namespace

int launch_dense_m128(const ssba_desc& d, float scale, const void* Q, const void* K, const void* V, void* O,
                      float* lse, cudaStream_t st)
{
    const long long N = (long long)d.H_tok * d.W_tok;
    const int BH = d.B * d.heads;
    if (d.head_dim != kD || d.dtype != SSBA_BF16 || N % kTile != 0 || N >= (1LL << 30)) return SSBA_ERR_UNSUPPORTED;
    DenseMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (!encode_tile_map(&maps.q, Q, BH, (int)N) || !encode_tile_map(&maps.k, K, BH, (int)N) ||
        !encode_tile_map(&maps.v, V, BH, (int)N)) {
        set_error("ssba_forward_dense: cuTensorMapEncodeTiled failed");
        return SSBA_ERR_CUDA;
    }
    DenseParams p;
    p.O = static_cast<__nv_bfloat16*>(O);
    p.lse = lse;
    p.BH = BH;
    p.N = (int)N;
    p.nt = (int)(N / kTile);
    p.units = BH * p.nt;
    p.scale_log2 = scale * 1.4426950408889634f;
    p.status = device_status_word();
    p.budget_ns = kWaitBudgetNs;
    if (!p.status) {
        set_error("ssba_forward_dense: could not resolve the device status word");
        return SSBA_ERR_CUDA;
    }
    const size_t smem = sizeof(DenseSmem) + 1024;
    g_dense_attr.run([smem] {
        cudaFuncSetAttribute(ssba_dense_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    const int want = (p.units + kStreams - 1) / kStreams;
    const int sms = device_sm_count();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(want < sms ? want : sms, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, ssba_dense_tc_kernel, maps, p);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("ssba_dense_tc_kernel launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

}  // namespace ssba
