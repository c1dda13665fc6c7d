// attn_tc.cu -- bf16 block-sparse attention forward on the sm_103a tensor cores
// (Sec. 2.2 "Efficient Sparse Execution": the kernel skips pruned blocks in its loads
// and its MMAs; Algorithm 1 SparseAttention over image tokens).
//
// Work item = one query block (64 tokens, an 8x8 window of the shifted grid) of one
// (batch, head); it visits only the key blocks listed for it. Two items are worked on at a
// time, as the two halves (rows 0-63 and 64-127) of M=128 products: half A is one item, half B
// another one, each with its own key blocks. Step t takes the t-th listed block of both:
//   S = [Q_A; Q_B] [K_A,t; K_B,t]^T   M=128 N=128 K=16 x 4: rows 0-63 need columns 0-63 of it,
//                                     rows 64-127 columns 64-127; the rest is never read
//   O_A += P_A V_A,t, O_B += P_B V_B,t   M=128 N=64 K=16, 4 + 4 products on the same O columns,
//                                     each with the other half's lanes masked off, so that
//                                     nothing of one item (an infinity, a NaN) reaches the other
// The products of a step cost what two M=64 products of each kind would, but the pair has one
// hand-off where two tiles had two, and a softmax thread owns a whole row of 64 scores. An item
// left over at the end of a pipeline's work takes both halves: the first half of its list in A,
// the second in B, merged at the end (two partial softmax sums).
// What bounds it: a step of each of the CTA's two pipelines takes 1430 (long lists) to 1600 cycles, of which the
// tensor pipe is busy 2 x 608 (QK 4 x 80, PV 8 x 36) and the softmax needs 2 x 435 of its scheduler;
// the rest is hand-offs (mbarrier waits, tensor-memory round trips) that two chains do not quite
// cover. Forward on given lists, 24 heads, GPU time in a graph of distinct layers, against the kernel with one
// 64-row tile per product: 4K (128 of 510 blocks) 2400 -> 1770 us, 2048 px (41 of 256) 400 -> 319, four 1024
// px images (16 of 64) 171 -> 150, one (11 of 64) 39.1 -> 35.8, 512 px (3 of 16) 10.6 -> 10.2. Where there is
// about one block for each of the 304 pipelines and a list is short, the longer step and the merge show: 288
// blocks of 3 8.1 -> 8.5 us.
// Persistent CTAs, one per SM (its 226 KB of shared memory fills the SM), each running two
// independent pipelines of 8 warps (512 threads, 128 registers each), warp-specialised:
//   K producer  (TMA, one lane). Q of each item and K, V of each listed key block arrive as 8 KB tiles
//               cut from [B*heads, H, W, d] tensor maps (128-byte swizzle): one 8x8-token box when the
//               shifted window does not cross the grid edge, else two or four boxes. A half-block
//               shift is a multiple of 4 tokens, so a crossing window splits 4 + 4: no gather pass
//               and no out-of-range fill. K and V have rings of three 16 KB stages each, Q one (the
//               next round's Q arrives while the softmax works on the last scores of this one).
//   QK issuer   QK of step t + 1 goes out as soon as the softmax holds S_t in registers and PV of
//               step t - 1 is done.
//   V producer  as the K producer, for the V ring.
//   PV issuer   PV of step t once P_t is stored and V_t has landed.
//   softmax     four warps, one TMEM lane quadrant each (two for half A, two for half B), one thread
//               per row. Online softmax in fp32 with exp2 in the log2-scaled domain against a
//               reference max m: the first step's row maximum. Later steps form P against it at once
//               and look at their row sum afterwards; only where that exceeds 2^24 (or is no number)
//               is the step's maximum taken, m raised, O rescaled in TMEM and P formed again. They
//               also write the finished items: O / l in bf16 and lse, after the exps of the next
//               item's first step, so that the wait for the item's last PV is spent on them.
// TMEM of a pipeline: S 128 + P 2 x 32 (bf16 pairs) + O 64 = 256 columns.
// In-kernel selection (ssba_forward_select): given the block means, each CTA first computes
// the score rows and the Top-k gating of its own items (one warp per item, the arithmetic of
// the mask kernels) and writes the lists to the caller's kv_idx / kv_cnt, which its producers
// then read back (coherent loads); no separate selection launch and no cross-CTA dependency.
// Tile rows follow the TMA box order of the window (tile_row_pos). All mbarrier waits are
// bounded (globaltimer budget + CTA abort flag); a timeout is reported in the device status
// word and the CTA drains its in-flight copies and MMAs before it exits.
#include <cuda.h>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "common.cuh"
#include "ptx.cuh"
#include "select.cuh"
#include "window.cuh"

namespace ssba {

namespace {

using namespace ptx;
using namespace win;

constexpr int kD = 64;
constexpr int kRows = 64;    // query rows per item = tokens per block
constexpr int kStages = 3;   // K ring, V ring
constexpr int kSlots = 2;                     // independent pipelines per CTA
constexpr int kSoftWarps = 4;                 // softmax warps of one pipeline
constexpr int kRoleWarps = 4;                 // K producer, QK issuer, V producer, PV issuer of one pipeline
constexpr int kThreads = kSlots * (kSoftWarps + kRoleWarps) * 32;
enum Role { kLoadK = 0, kQK = 1, kLoadV = 2, kPV = 3, kSoftmax = 4 };
constexpr uint32_t kSlotCols = 256;           // TMEM columns of one pipeline
constexpr uint32_t kTmemCols = kSlots * kSlotCols;
constexpr uint32_t kColS = 0;    // S: [0,128)
constexpr uint32_t kColP = 128;  // P buffers: [128,160), [160,192)
constexpr uint32_t kColO = 192;  // O accumulator: [192,256)
constexpr uint32_t kTileBytes = kRows * kD * 2;    // 8 KB: one block of one tensor
constexpr uint32_t kPairBytes = 2 * kTileBytes;    // both halves
// A step's row sum of exp2(s c - m) above which the row's reference max m is raised. Any value would
// give the same precision (P, O and l are floating-point numbers, of any common scale); this one
// leaves O 2^100 of head room over V, and a later step has to exceed the first one's maximum by
// 2^18 to reach it.
constexpr float kRaise = 16777216.f;  // 2^24
constexpr int kCntCap = 40;  // item counts of a pipeline held in shared memory (20 rounds)

// QK: M=128, A (Q) and B (K) K-major; N=64 in a step that only one half takes part in. PV: M=128
// N=64, A (P) K-major, B (V) MN-major.
constexpr uint32_t kIdescQK = idesc_bf16_f32(128, 128, false, false);
constexpr uint32_t kIdescQK1 = idesc_bf16_f32(128, 64, false, false);
constexpr uint32_t kIdescPV = idesc_bf16_f32(128, 64, false, true);

struct __align__(1024) SlotSmem {
    uint8_t k[kStages][kPairBytes];
    uint8_t v[kStages][kPairBytes];
    uint8_t q[kPairBytes];
};

// Barriers and schedule of one pipeline.
struct SlotCtl {
    uint64_t k_full[kStages];
    uint64_t k_empty[kStages];
    uint64_t v_full[kStages];
    uint64_t v_empty[kStages];
    uint64_t q_full;
    uint64_t q_empty;
    uint64_t s_full;      // QK_g has finished
    uint64_t s_free;      // the four softmax warps hold S_g in registers
    uint64_t p_full[2];   // the four softmax warps have stored P_g (and read the last item's O); two, as
                          // they may store P_{g+1} before the issuer, waiting for V_g, sees P_g
    uint64_t o_full[2];   // PV_g has finished
    uint64_t merged;      // half B's part of a split item is in shared memory
    uint64_t drain[2];
    int32_t cnts[kCntCap];  // counts of the first items, in walk order
    int first, stride, last, rounds, single;  // see build_schedule
};

constexpr int kWinCap = 256;  // labels whose window (origin, box shape) is tabulated per CTA (2048 px: 256)

// Timeline instrumentation, compiled only into the timeline build of the library (-DSSBA_TIMELINE;
// the default build has none of it). Per CTA, globaltimer stamps (ns) of the launch's phases; per
// step of eight sampled pipelines (pipeline 0 and 1 of CTAs 0, 1, gridDim/2 and gridDim-1), SM
// clock stamps of each role, and per round those of the finished rows. ssba_timeline_read copies them out.
namespace tl {
constexpr int kCtas = 256, kCtaEv = 16, kPipes = 4 * kSlots, kTiles = 128, kTileEv = 10, kItems = 32, kItemEv = 4;
enum CtaEv { kEntry = 0, kDepWait, kPoolLanded, kPooled, kBarrier, kStaged, kSelected, kPipesStart, kSlot0End,
             kSlot1End, kEnd, kSelStart, kScoresDone, kWalkDone };
// step events: K copy issued, QK issued, softmax saw S, softmax done with the exps, P stored, PV
// issued, V copy issued, QK's waits over, S in the softmax's registers, PV's waits over (the
// softmax's of half A's first warp)
enum TileEv { kKIssue = 0, kQKIssue, kSmxStart, kSmxExp, kPStored, kPVIssue, kVIssue, kSFree, kSLoaded, kPVReady };
// round events: half A's rows are due (their wait for the last PV starts), O ready, rows written
enum ItemEv { kEpiStart = 0, kEpiO, kEpiDone, kPipeClock0 };
#ifdef SSBA_TIMELINE
__device__ unsigned long long cta_ev[kCtas][kCtaEv];
__device__ unsigned int tile_ev[kPipes][kTiles][kTileEv];
__device__ unsigned int item_ev[kPipes][kItems][kItemEv];
__device__ __forceinline__ int pipe_of(int slot)
{
    const int b = blockIdx.x, G = gridDim.x;
    const int s = b == 0 ? 0 : (b == 1 ? 1 : (b == G / 2 ? 2 : (b == G - 1 ? 3 : -1)));
    return s < 0 ? -1 : s * kSlots + slot;
}
#endif
}  // namespace tl
// -DSSBA_TIMELINE=1 records the per-CTA phase stamps only (they barely perturb the launch);
// -DSSBA_TIMELINE=2 also the per-tile and per-item stamps of the sampled pipelines.
#ifdef SSBA_TIMELINE
#define TL_CTA(ev)                                                                              \
    do {                                                                                        \
        if (blockIdx.x < tl::kCtas) tl::cta_ev[blockIdx.x][ev] = ptx::globaltimer_ns();        \
    } while (0)
#if SSBA_TIMELINE >= 2
#define TL_TILE(slot, gb, ev)                                                                   \
    do {                                                                                        \
        const int tl_p_ = tl::pipe_of(slot);                                                    \
        if (tl_p_ >= 0 && (gb) < (uint32_t)tl::kTiles) tl::tile_ev[tl_p_][gb][ev] = (unsigned)clock(); \
    } while (0)
#define TL_ITEM(slot, n, ev)                                                                    \
    do {                                                                                        \
        const int tl_p_ = tl::pipe_of(slot);                                                    \
        if (tl_p_ >= 0 && (n) < (uint32_t)tl::kItems) tl::item_ev[tl_p_][n][ev] = (unsigned)clock(); \
    } while (0)
#else
#define TL_TILE(slot, gb, ev) do { } while (0)
#define TL_ITEM(slot, n, ev) do { } while (0)
#endif
#else
#define TL_CTA(ev) do { } while (0)
#define TL_TILE(slot, gb, ev) do { } while (0)
#define TL_ITEM(slot, n, ev) do { } while (0)
#endif

constexpr int kPoolUnits = 2 * (2 * kStages + 1);  // 8 KB pooling buffers of one pipeline's stages

struct __align__(1024) SmemLayout {
    SlotSmem slot[kSlots];
    SlotCtl ctl[kSlots];
    uint32_t win[kWinCap];  // label -> r0 | c0 << 15 | box shape << 30 (see window_entry)
    uint64_t pool_bar[kSlots * kPoolUnits];  // one per buffer: its block's rows landed (in-kernel pooling)
    uint32_t tmem_base;
    int abort_flag;
};

// Four maps per tensor, one per box shape, over the [B*heads][H][W][d] bf16 view, and
// the text keys and values as [B*heads][T_txt][d] (64-row boxes, zero fill past T_txt).
static_assert(sizeof(SmemLayout) + 1024 <= 232448, "shared memory of one CTA (227 KB opt-in limit)");
static_assert(sizeof(SlotSmem) == kPoolUnits * kTileBytes, "stages back to back");

struct TileMaps {
    CUtensorMap q[4], k[4], v[4];
    CUtensorMap kt, vt;
};

struct TcParams {
    __nv_bfloat16* O;
    float* lse;
    const int32_t* idx;  // null: dense mode, every block of the head
    const int32_t* cnt;
    Grid g;
    int keep;          // length of an index-list row
    int ntxt;          // text key blocks visited first by every query block (ceil(T_txt / 64))
    int t_txt;         // text tokens
    int units;         // key blocks of a whole item: ntxt + keep
    int num_items;
    float scale_log2;  // softmax scale * log2(e)
    int* status;       // device status word
    const float* sel_qb;  // in-kernel selection: block means [B*heads][Tb][64] (null: lists given)
    const float* sel_kb;
    int32_t* sel_cnt;     // counts written by the selection
    float* sel_scores;    // optional S export [B*heads][Tb][Tb]
    // in-kernel pooling (ssba_forward_fused): the warps of the grid pool the (block, tensor)
    // units into sel_qb / sel_kb, then the CTAs meet at a grid barrier (null: means given)
    const __nv_bfloat16* pool_q;
    const __nv_bfloat16* pool_k;
    unsigned* gsync;  // grid barrier words in the workspace (arrivals, departures)
    uint64_t budget_ns;  // wall-time limit of every barrier wait
    int withhold;        // failure-detection test hooks: 1, pipeline 0 announces its first K copy
                         // but never issues it, so that the waits on it run out; 2, CTA 0 does not
                         // arrive at the grid barrier of the fused launch (0 otherwise)
};

// Work schedule, for V pipelines (two per CTA): each takes its items two at a time (a round), a
// single one left over alone, split over the two halves.
//   Lists given: neighbouring items form a pair, pairs go round-robin (neighbouring pipelines work
//     on neighbouring items, so the K/V tiles of a few heads are shared through L2); of the items
//     left after the whole rounds each pipeline takes one, or the first ones a pair.
//   In-kernel selection: contiguous ranges (item counts differing by at most one), so that the
//     few items of a CTA share one or two heads and the selection stages each head's k_b once.
// Pipeline `slot` of CTA b is number b + slot * CTAs: the longer shares go to different CTAs.
__device__ __forceinline__ int sel_item_count(const TcParams& p, int v, int V)
{
    return p.num_items / V + (v < p.num_items % V ? 1 : 0);
}
__device__ __forceinline__ int sel_first_item(const TcParams& p, int v, int V)
{
    return v * (p.num_items / V) + min(v, p.num_items % V);
}

// One round: per half the item, the first block (position in the item's blocks, text first) and
// the number of blocks.
struct Round {
    int item[2], tb[2], nb[2];
    bool split;  // both halves work on the same item
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
    uint64_t t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity))
        if (globaltimer_ns() - t0 > budget_ns) return false;
    return true;
}

__device__ __forceinline__ int clamp_label(int j, int Tb) { return j < 0 ? 0 : (j >= Tb ? Tb - 1 : j); }

// Checked build (-DSSBA_CHECKED, build.py variant "checked"): the invariants of the index lists
// the kernel reads (every label in [0, Tb), each row strictly ascending, every count in [0, keep])
// are tested, and a violation is reported as SSBA_ERR_CHECK in the device status word; the value
// is still clamped as in the default build, which tests nothing.
#ifdef SSBA_CHECKED
constexpr bool kChecked = true;
#else
constexpr bool kChecked = false;
#endif

// Block means of the whole layer inside the launch: unit u is (tensor u & 1, item u >> 1); the
// CTA takes the units u = i gridDim + blockIdx, i < kSlots * kPoolUnits at a time, one 8 KB piece
// of the idle stage buffers each, warp w units w and w + 16 of them (all copies of a batch in
// flight together). Lanes 0..7 bulk-copy the unit's eight token rows (one copy per row, two where
// the shifted window wraps the right edge), and after the copies land every lane sums its (row
// group, column chunk) with the loop order of ssba_pool_blocks_kernel, so the means are those of
// ssba_pool_blocks bit for bit. Returns false if a copy did not land in time (after a second
// bounded wait for it).
__device__ __noinline__ bool pool_phase(const TcParams& p, SmemLayout& cs, int gwarp, int lane, volatile int* abortf)
{
    constexpr int VE = 8, CPR = kD / VE, RPI = 32 / CPR, LOADS = 64 / RPI;
    constexpr int kWarps = kThreads / 32, kUnits = kSlots * kPoolUnits;
    const Grid& g = p.g;
    const int Tb = g.Tb(), N = g.H * g.W;
    const int col = lane % CPR, r0 = lane / CPR;
    const int total = 2 * p.num_items;
    int round = 0;
    for (int base = 0; base * (int)gridDim.x + (int)blockIdx.x < total; base += kUnits, ++round) {
        for (int q = gwarp; q < kUnits; q += kWarps) {
            const int u = (base + q) * gridDim.x + blockIdx.x;
            if (u >= total) break;
            const uint32_t bar = smem_u32(&cs.pool_bar[q]);
            const uint32_t buf = smem_u32(&cs.slot[q / kPoolUnits].k[0][0]) + (q % kPoolUnits) * kTileBytes;
            const int which = u & 1, item = u >> 1;
            const int bh = item / Tb, label = item - bh * Tb;
            const int br = label / g.bw, bc = label - br * g.bw;
            const int rb = br * 8 - g.sr, cb = bc * 8 - g.sc;
            if (round > 0) {
                __syncwarp();
                fence_proxy_async_smem();  // the last round's reads before the copies overwrite them
            }
            if (lane == 0) mbar_arrive_expect_tx(bar, kTileBytes);
            __syncwarp();
            if (lane < 8) {
                const __nv_bfloat16* X = (which ? p.pool_k : p.pool_q) + (size_t)bh * N * kD;
                int r = rb + lane;
                r += r < 0 ? g.H : 0;
                const uint32_t dst = buf + lane * 8 * kD * 2;
                // columns cb .. cb + 7 with -W < cb <= W - 8, each negative one taken + W
                if (cb >= 0 || cb <= -8) {  // one run of 8 columns
                    bulk_load(dst, X + (size_t)(r * g.W + (cb < 0 ? cb + g.W : cb)) * kD, 8 * kD * 2, bar);
                } else {  // columns W + cb .. W - 1, then 0 .. 7 + cb
                    const int n1 = -cb;  // 1 .. 7
                    bulk_load(dst, X + (size_t)(r * g.W + g.W + cb) * kD, n1 * kD * 2, bar);
                    bulk_load(dst + n1 * kD * 2, X + (size_t)r * g.W * kD, (8 - n1) * kD * 2, bar);
                }
            }
        }
        for (int q = gwarp; q < kUnits; q += kWarps) {
            const int u = (base + q) * gridDim.x + blockIdx.x;
            if (u >= total) break;
            const uint32_t bar = smem_u32(&cs.pool_bar[q]);
            const uint8_t* buf = &cs.slot[q / kPoolUnits].k[0][0] + (q % kPoolUnits) * kTileBytes;
            const int which = u & 1, item = u >> 1;
            if (!mbar_wait(bar, round & 1, abortf, p.budget_ns)) {
                volatile int never = 0;  // wait once more, for the copies only, before giving up
                for (int x = gwarp; x < kUnits && (base + x) * (int)gridDim.x + (int)blockIdx.x < total; x += kWarps)
                    mbar_wait(smem_u32(&cs.pool_bar[x]), round & 1, &never, p.budget_ns);
                return false;
            }
            if (gwarp == 0 && lane == 0 && round == 0 && q == 0) TL_CTA(tl::kPoolLanded);
            float acc[VE];
#pragma unroll
            for (int e = 0; e < VE; ++e) acc[e] = 0.f;
#pragma unroll
            for (int i = 0; i < LOADS; ++i) {
                const int pos = r0 + i * RPI;
                const uint4 v = *reinterpret_cast<const uint4*>(buf + (pos * kD + col * VE) * 2);
                const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 f = __bfloat1622float2(h2[e]);
                    acc[2 * e] += f.x;
                    acc[2 * e + 1] += f.y;
                }
            }
#pragma unroll
            for (int o = CPR; o < 32; o <<= 1)
#pragma unroll
                for (int e = 0; e < VE; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
            if (r0 == 0) {
                float* dst = const_cast<float*>(which ? p.sel_kb : p.sel_qb) + (size_t)item * kD + col * VE;
                constexpr float kInv = 1.0f / 64.0f;
                reinterpret_cast<float4*>(dst)[0] = make_float4(acc[0] * kInv, acc[1] * kInv, acc[2] * kInv, acc[3] * kInv);
                reinterpret_cast<float4*>(dst)[1] = make_float4(acc[4] * kInv, acc[5] * kInv, acc[6] * kInv, acc[7] * kInv);
            }
        }
    }
    return true;
}

// Grid-wide barrier for a persistent launch whose CTAs are all resident (one per SM, grid at
// most the SM count; the next grid is released only after it). Called by one thread of each
// CTA after a CTA barrier: a release add makes the CTA's writes (ordered before it by that
// barrier) visible with its arrival, and an acquire load sees every other CTA's. w[0] counts
// arrivals; the reset is left to grid_barrier_depart at the end of the kernel, off the
// critical path. Bounded; returns false on timeout or abort.
__device__ bool grid_barrier_arrive_wait(unsigned* w, unsigned n, volatile int* abortf, uint64_t budget_ns,
                                         bool arrive)
{
    if (arrive) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(w) : "memory");
    const uint64_t t0 = globaltimer_ns();
    for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(w) : "memory");
        if (v == n) return true;
        if (*abortf || globaltimer_ns() - t0 > budget_ns) return false;
    }
}

// After a CTA has passed the barrier: w[1] counts departures, and the last CTA to pass sets both words
// back to zero (nobody polls them any more), so a call that completes leaves the workspace
// zero-filled. The count is taken at once and its answer looked at later (grid_barrier_reset): the
// round trip of the atomic is off the launch's critical path, where at the end of the kernel it
// added about a microsecond. (A CTA that gave up at the barrier does not depart; the workspace is
// then zeroed again by the caller, as after any timeout.)
__device__ __forceinline__ unsigned grid_barrier_depart(unsigned* w) { return atomicAdd(&w[1], 1u); }
__device__ __forceinline__ void grid_barrier_reset(unsigned* w, unsigned n, unsigned departed)
{
    if (departed == n - 1) {
        atomicExch(&w[0], 0u);
        atomicExch(&w[1], 0u);
    }
}

// A list entry: written earlier in this launch under in-kernel selection (read through L2),
// else read-only input.
template <bool kSel>
__device__ __forceinline__ int ld_list(const int32_t* a) { return kSel ? __ldcg(a) : __ldg(a); }

// Score row and Top-k gating of one item (one warp), with the arithmetic and the selection code
// of the mask kernels (S_j = q_b . k_b[j], four interleaved partial sums over d combined in a
// fixed order; sel::ballot_select on keys held in registers), so the same means give the same lists.
// kbs: the head's k_b
// staged in shared memory, the 16-byte chunk c4 of row j at chunk c4 ^ (j & 15) (two lanes per
// bank at most when 32 lanes read one column); qs: the item's q_b row in shared memory. Not
// inlined, so that its registers do not weigh on the pipeline roles.
template <int kPer>
__device__ __noinline__ void select_item(const TcParams& p, int item, int lane, const float* kbs, const float* qs)
{
    const int Tb = p.g.Tb();
    const bool stamp = threadIdx.x == 0 && item == sel_first_item(p, blockIdx.x, gridDim.x * kSlots);
    if (stamp) TL_CTA(tl::kSelStart);
    uint32_t key[kPer];
#pragma unroll
    for (int m = 0; m < kPer; ++m) {
        const int j = lane + 32 * m;
        key[m] = 0u;
        if (j < Tb) {
            const float* row = kbs + j * kD;
            float s1[1];
            sel::affinity<1>(s1, qs, kD, [&](int c) { return *reinterpret_cast<const float4*>(row + 4 * (c ^ (j & 15))); });
            const float acc = s1[0];
            if (p.sel_scores) p.sel_scores[(size_t)item * Tb + j] = acc;
            key[m] = sel::order_key(acc);
        }
    }
    if (stamp) TL_CTA(tl::kScoresDone);
    sel::ballot_select<kPer>(key, Tb, p.keep, lane, const_cast<int32_t*>(p.idx) + (size_t)item * p.keep);
    if (stamp) TL_CTA(tl::kWalkDone);
    if (lane == 0) p.sel_cnt[item] = p.keep;
    __syncwarp();
}

// Round r of a pipeline from its schedule in shared memory.
template <bool kSel>
__device__ __forceinline__ Round get_round(const TcParams& p, const SlotCtl& c, int r)
{
    Round rd;
    const bool end = r == c.rounds - 1;
    rd.split = end && c.single;
    rd.item[0] = end ? c.last : c.first + r * c.stride;
    rd.item[1] = rd.item[0] + (rd.split ? 0 : 1);
    rd.tb[0] = rd.tb[1] = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        int n = p.units;
        if (!kSel && p.idx)
            n = p.ntxt + (2 * r + h < kCntCap ? c.cnts[2 * r + h] : min(max(__ldg(p.cnt + rd.item[h]), 0), p.keep));
        rd.nb[h] = n;
    }
    if (rd.split) {
        rd.tb[1] = (rd.nb[0] + 1) >> 1;
        rd.nb[1] = rd.nb[0] - rd.tb[1];
        rd.nb[0] = rd.tb[1];
    }
    return rd;
}

// Fills the schedule of pipeline v (thread t of its nthr threads); see the work-schedule
// comment above. Rounds r < rounds - 1 are the pairs of items first + r stride, + 1; the last one
// is the pair (or, single set, the one item) at `last`.
template <bool kSel>
__device__ __forceinline__ void build_schedule(const TcParams& p, SlotCtl& c, int v, int V, int t, int nthr)
{
    int first, stride, last, rounds, single;
    if (kSel) {
        const int n = sel_item_count(p, v, V);
        first = sel_first_item(p, v, V);
        stride = 2;
        rounds = (n + 1) / 2;
        single = n & 1;
        last = first + 2 * (rounds - 1);
    } else {
        const int full = p.num_items / (2 * V), base = full * 2 * V, rem = p.num_items - base;
        const int pairs = max(0, rem - V);  // pipelines that take a pair of the rest, the others one item
        const int n = v < pairs ? 2 : (v < rem ? 1 : 0);
        first = 2 * v;
        stride = 2 * V;
        rounds = full + (n > 0);
        single = n == 1;
        last = n > 0 ? base + v + min(v, pairs) : first + (full - 1) * stride;
    }
    if (!kSel && p.idx)
        for (int i = t; i < 2 * rounds && i < kCntCap; i += nthr) {
            const int r = i >> 1, item = (r == rounds - 1 ? last : first + r * stride) + (i & 1);
            if (item < p.num_items) c.cnts[i] = min(max(__ldg(p.cnt + item), 0), p.keep);
        }
    if (t != 0) return;
    c.first = first;
    c.stride = stride;
    c.last = last;
    c.rounds = rounds;
    c.single = single;
}

// D[tmem] (+)= A[tmem] * B[smem]^T on half h's 64 lanes only: the other lanes of D keep their value.
__device__ __forceinline__ void mma_ts_half(int h, uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate)
{
    const uint32_t off_a = h ? 0xffffffffu : 0u, off_b = ~off_a;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %5, %6, %6}, p;\n"
        "}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(off_a), "r"(off_b)
        : "memory");
}

// Row of a finished item: O / l in bf16 and lse to global memory, O (unnormalised) read from TMEM
// in two chunks, the other part of a split item (b_o: its row in shared memory, 16-byte chunks
// swizzled by row) added with weights wa, wb first. A part whose a_ok, b_ok is false has a sum of 0 and
// counts for nothing; a weight that vanishes does not drop its part, so that an infinity or NaN of V
// under it comes out as it does where O is rescaled within one half.
__device__ __forceinline__ void store_row(const TcParams& p, int item, int row, uint32_t ocol, float m, float l,
                                          const float* b_o = nullptr, float wa = 1.f, float wb = 0.f,
                                          bool a_ok = true, bool b_ok = false)
{
    const int Tb = p.g.Tb(), N = p.g.H * p.g.W;
    const int bh = item / Tb, label = item - bh * Tb;
    const bool ok = l > 0.f;
    const float inv = ok ? 1.f / l : 0.f;
    const int tok = p.g.token(label, tile_row_pos(p.g, label, row));
    uint4* dst = reinterpret_cast<uint4*>(p.O + ((size_t)bh * N + tok) * kD);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t o[32];
        tmem_ld_32x32b_x32(ocol + 32 * c, o);
        tmem_wait_ld();
        if (b_o) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 x = *reinterpret_cast<const float4*>(b_o + 4 * ((8 * c + i) ^ (row & 15)));
                const float xb[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float a = a_ok ? __uint_as_float(o[4 * i + e]) * wa : 0.f;
                    o[4 * i + e] = __float_as_uint(b_ok ? fmaf(xb[e], wb, a) : a);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = ok ? __uint_as_float(o[8 * i + e]) * inv : 0.f;
            dst[4 * c + i] = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]),
                                        pack_bf16(f[6], f[7]));
        }
    }
    p.lse[(size_t)bh * N + tok] = ok ? (m * 0.69314718055994531f + logf(l)) : -INFINITY;
}

// kSel: the lists are selected here, from means given or (p.pool_q) pooled here too; without it they are
// given. Two kernels, so that the set-up of the one costs the pipelines of the other nothing: the
// registers and the code of the whole kernel move with every edit of it (7 % of the forward on given
// lists, measured, for a change inside select_item).
template <bool kSel>
__global__ void __launch_bounds__(kThreads, 1) ssba_attn_tc_kernel(const __grid_constant__ TileMaps maps,
                                                                   const TcParams p)
{
    extern __shared__ uint8_t smem_raw[];
    SmemLayout& cs = *reinterpret_cast<SmemLayout*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                    ~static_cast<uintptr_t>(1023));
    const int gwarp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) TL_CTA(tl::kEntry);
    if (threadIdx.x < kSlots * kSoftWarps * 32 && threadIdx.x % (kSoftWarps * 32) == 0) {
        const int slot = threadIdx.x / (kSoftWarps * 32);
        SlotCtl& sm = cs.ctl[slot];
        if (slot == 0) cs.abort_flag = 0;
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&sm.k_full[s]), 1);
            mbar_init(smem_u32(&sm.k_empty[s]), 1);
            mbar_init(smem_u32(&sm.v_full[s]), 1);
            mbar_init(smem_u32(&sm.v_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&sm.p_full[b]), 4);
            mbar_init(smem_u32(&sm.o_full[b]), 1);
            mbar_init(smem_u32(&sm.drain[b]), 1);
        }
        mbar_init(smem_u32(&sm.q_full), 1);
        mbar_init(smem_u32(&sm.q_empty), 1);
        mbar_init(smem_u32(&sm.s_full), 1);
        mbar_init(smem_u32(&sm.s_free), 4);
        mbar_init(smem_u32(&sm.merged), 2);
        if (kSel && p.pool_q)
            for (int w = slot * kPoolUnits; w < (slot + 1) * kPoolUnits; ++w) mbar_init(smem_u32(&cs.pool_bar[w]), 1);
        fence_mbar_init();
    }
    for (int l = threadIdx.x; l < p.g.Tb() && l < kWinCap; l += kThreads) cs.win[l] = window_entry(p.g, l);
    if (gwarp == 2 && lane < 12) tma_prefetch_desc(lane < 4 ? &maps.q[lane] : (lane < 8 ? &maps.k[lane - 4] : &maps.v[lane - 8]));
    if (gwarp == 1) {
        tmem_alloc(smem_u32(&cs.tmem_base), kTmemCols);
        tmem_relinquish();
    }
    // everything above reads no input; the lists, counts and tensors may come from the grid
    // launched just before this one (programmatic dependent launch)
    grid_dep_wait();
    if (threadIdx.x == 0) TL_CTA(tl::kDepWait);
    bool pool_fail = false;
    unsigned departed = 0;
    if (kSel && p.pool_q) {
        // the block means of the whole layer, the (block, tensor) units shared out over the grid,
        // then a grid barrier; the next grid is released only after it, so that it cannot take
        // an SM that one of these CTAs still waits for
        __syncthreads();  // the pooling barriers are initialised
        pool_fail = !pool_phase(p, cs, gwarp, lane, &cs.abort_flag);
        pool_fail = __syncthreads_or(pool_fail);  // also orders this CTA's means before the arrival
        if (threadIdx.x == 0) TL_CTA(tl::kPooled);
        if (threadIdx.x == 0 && !pool_fail)
            pool_fail = !grid_barrier_arrive_wait(p.gsync, gridDim.x, &cs.abort_flag, p.budget_ns,
                                                  p.withhold != 2 || blockIdx.x != 0);
        // on a timeout the means of other CTAs may be missing: the status is set, and the raised
        // abort flag makes every role leave at its first wait that does not complete at once
        // (lists selected from stale means still hold labels in [0, Tb))
        pool_fail = __syncthreads_or(pool_fail);
        if (threadIdx.x == 0) TL_CTA(tl::kBarrier);
        if (threadIdx.x == 0) {
            if (pool_fail) {
                atomicExch(p.status, SSBA_ERR_TIMEOUT);
                cs.abort_flag = 1;
            } else {
                departed = grid_barrier_depart(p.gsync);
            }
        }
    }
    grid_dep_launch();
    // which pipeline of this CTA, and the role within it: the softmax warps first, so that a
    // pipeline's four are one per TMEM lane quadrant (and two softmax warps share a scheduler)
    const bool soft = gwarp < kSlots * kSoftWarps;
    const int slot = soft ? gwarp / kSoftWarps : (gwarp - kSlots * kSoftWarps) / kRoleWarps;
    const int role = soft ? kSoftmax : (gwarp - kSlots * kSoftWarps) % kRoleWarps;
    SlotSmem& sm = cs.slot[slot];
    SlotCtl& ct = cs.ctl[slot];
    volatile int* abortf = &cs.abort_flag;
    const int vcta = slot * gridDim.x + blockIdx.x;
    const int vgrid = gridDim.x * kSlots;
    const int Tb = p.g.Tb();
    if (kSel) {
        // the lists of this CTA's items (the contiguous ranges of its two pipelines): the k_b
        // of the heads they touch are staged by all threads in the stage buffers of both
        // pipelines (free until the producers start), one asynchronous round per batch of
        // heads; then one warp per item
        const int f0 = sel_first_item(p, blockIdx.x, vgrid), n0 = sel_item_count(p, blockIdx.x, vgrid);
        const int f1 = sel_first_item(p, blockIdx.x + gridDim.x, vgrid);
        const int n1 = sel_item_count(p, blockIdx.x + gridDim.x, vgrid);
        // heads of the two ranges: [h0a, h0b] and [h1a, h1b], staged in that order
        const int h0a = f0 / Tb, h0b = n0 ? (f0 + n0 - 1) / Tb : h0a - 1;
        const int h1a = f1 / Tb, h1b = n1 ? (f1 + n1 - 1) / Tb : h1a - 1;
        const int nh0 = max(0, h0b - h0a + 1), nh = nh0 + max(0, h1b - h1a + 1);
        auto head_of = [&](int hi) { return hi < nh0 ? h0a + hi : h1a + (hi - nh0); };
        // staging: pipeline 0's k, v, q buffers end with the scratch (a 64-float query row per warp, then
        // up to kSelQRows shared query rows, more than the kSelItems an SM of a call that selects here;
        // only the failure-detection hook can bring more); the rest of them and pipeline 1's hold the heads
        constexpr uint32_t kRegion = sizeof(SlotSmem);  // k, v, q of one pipeline
        constexpr int kSelQRows = 24;
        constexpr uint32_t kScratch = (kThreads / 32 + kSelQRows) * kD * 4;
        const uint32_t hb = (uint32_t)Tb * kD * 4;
        const int cap0 = (int)((kRegion - kScratch) / hb), cap = cap0 + (int)(kRegion / hb);
        uint8_t* r0 = &cs.slot[0].k[0][0];
        float* own = reinterpret_cast<float*>(r0 + kRegion - kScratch) + gwarp * kD;
        float* qrows = reinterpret_cast<float*>(r0 + kRegion - kScratch) + (kThreads / 32) * kD;
        auto staged = [&](int hi) {
            return reinterpret_cast<float*>(hi < cap0 ? r0 + hi * hb : &cs.slot[1].k[0][0] + (hi - cap0) * hb);
        };
        auto item_of = [&](int q) { return q < n0 ? f0 + q : f1 + (q - n0); };
        for (int base = 0; base < nh; base += cap) {
            const int m = min(cap, nh - base);
            // asynchronous 16-byte copies, all in flight at once: the heads' k_b (chunk c4 of row
            // j to chunk c4 ^ (j & 15)) and, in the first round, the items' q_b rows
            for (int e = threadIdx.x; e < m * Tb * (kD / 4); e += kThreads) {
                const int hi = e / (Tb * (kD / 4)), rem = e - hi * Tb * (kD / 4);
                const int j = rem / (kD / 4), c4 = rem - j * (kD / 4);
                const float* src = p.sel_kb + ((size_t)head_of(base + hi) * Tb + j) * kD + 4 * c4;
                const uint32_t dst = smem_u32(staged(hi) + j * kD + 4 * (c4 ^ (j & 15)));
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
            }
            if (base == 0)
                for (int e = threadIdx.x; e < min(n0 + n1, kSelQRows) * (kD / 4); e += kThreads) {
                    const int q = e / (kD / 4), c4 = e - q * (kD / 4);
                    const float* src = p.sel_qb + (size_t)item_of(q) * kD + 4 * c4;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(qrows + q * kD + 4 * c4)),
                                 "l"(src) : "memory");
                }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            if (threadIdx.x == 0 && base == 0) TL_CTA(tl::kStaged);
            // the items whose head is in this batch
            for (int q = gwarp; q < n0 + n1; q += kThreads / 32) {
                const int item = item_of(q);
                const int h = item / Tb;
                const int hi = (q < n0 ? h - h0a : nh0 + h - h1a) - base;
                if (hi < 0 || hi >= m) continue;
                const float* qs = qrows + q * kD;
                if (q >= kSelQRows) {  // rows past the staged ones: this warp's own copy
                    if (lane < kD / 4)
                        reinterpret_cast<float4*>(own)[lane] =
                            __ldcg(reinterpret_cast<const float4*>(p.sel_qb + (size_t)item * kD) + lane);
                    __syncwarp();
                    qs = own;
                }
                if (Tb <= 32) select_item<1>(p, item, lane, staged(hi), qs);
                else if (Tb <= 64) select_item<2>(p, item, lane, staged(hi), qs);
                else if (Tb <= 128) select_item<4>(p, item, lane, staged(hi), qs);
                else select_item<8>(p, item, lane, staged(hi), qs);
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) TL_CTA(tl::kSelected);
        if (p.pool_q && threadIdx.x == 0 && !pool_fail) grid_barrier_reset(p.gsync, gridDim.x, departed);
    }
    if (soft) build_schedule<kSel>(p, ct, vcta, vgrid, threadIdx.x % (kSoftWarps * 32), kSoftWarps * 32);
    // the stage buffers held the pooled rows and the staged means (generic accesses); the
    // producers' tensor copies (async proxy) overwrite them next
    if (kSel) fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = cs.tmem_base + slot * kSlotCols;
    const int rounds = ct.rounds;
    const uint32_t abort_at = smem_u32(&cs.abort_flag);
    bool dead = false;
    uint32_t g = 0;  // steps that the role is through with
    int nq = 0;      // (K producer) rounds whose Q is announced
    if (threadIdx.x == 0) TL_CTA(tl::kPipesStart);
    if (soft && threadIdx.x % (kSoftWarps * 32) == 0) TL_ITEM(slot, 0u, tl::kPipeClock0);

    if (role == kLoadK || role == kLoadV) {
        // ------------------------------------------------------------ TMA producers
        // The K producer loads each round's Q tiles and the K tiles of its key blocks, the V producer
        // the V tiles, one elected lane for both halves. A K stage frees when its QK is done and a V
        // stage when its PV is done, so the rings do not wait on each other. All lanes fetch the
        // labels of 32 steps at once and look up their windows; each step's two entries then come
        // from a shuffle.
        const bool is_k = role == kLoadK;
        const uint32_t empty0 = smem_u32(is_k ? &ct.k_empty[0] : &ct.v_empty[0]);
        const uint32_t full0 = smem_u32(is_k ? &ct.k_full[0] : &ct.v_full[0]);
        const uint32_t tile0 = smem_u32(is_k ? &sm.k[0][0] : &sm.v[0][0]);
        const CUtensorMap* m4 = is_k ? maps.k : maps.v;
        const CUtensorMap* mt = is_k ? &maps.kt : &maps.vt;
        // test hook: the first K copies of pipeline 0 never land
        const bool hold = p.withhold == 1 && is_k && vcta == 0;
        auto entry_of = [&](int label) { return label < kWinCap ? cs.win[label] : window_entry(p.g, label); };
        for (int r = 0; !dead && r < rounds; ++r) {
            const Round rd = get_round<kSel>(p, ct, r);
            const int steps = max(rd.nb[0], rd.nb[1]);
            const int bh0 = rd.item[0] / Tb, bh1 = rd.item[1] / Tb;
            if (kChecked && is_k && p.idx) {
                // the entries of both halves ascending and in range (the one before a second part
                // too), and the items' counts in [0, keep]
                bool bad = false;
                for (int h = 0; h < 2; ++h) {
                    const int32_t* hl = p.idx + (size_t)rd.item[h] * p.keep;
                    const int a = max(rd.tb[h], p.ntxt) - p.ntxt, b = rd.tb[h] + rd.nb[h] - p.ntxt;
                    for (int t = a + lane; t < b; t += 32) {
                        const int raw = ld_list<kSel>(hl + t);
                        bad |= raw < 0 || raw >= Tb;
                        if (t > 0) bad |= raw <= ld_list<kSel>(hl + t - 1);
                    }
                    if (lane == 0 && !kSel) {
                        const int c = __ldg(p.cnt + rd.item[h]);
                        bad |= c < 0 || c > p.keep;
                    }
                }
                if (__any_sync(0xffffffffu, bad) && lane == 0) atomicExch(p.status, SSBA_ERR_CHECK);
                __syncwarp();
            }
            // the round's Q pair, once the last round's final QK has read its own
            auto load_q = [&]() -> bool {
                const bool ok = mbar_wait(smem_u32(&ct.q_empty), (r & 1) ^ 1, abortf, p.budget_ns);
                if (!__all_sync(0xffffffffu, ok)) return false;
                if (elect_one_sync()) {
                    const uint32_t bar = smem_u32(&ct.q_full);
                    mbar_arrive_expect_tx(bar, kPairBytes);
                    window_boxes_e(maps.q, smem_u32(&sm.q[0]), bar, entry_of(rd.item[0] - bh0 * Tb), bh0);
                    window_boxes_e(maps.q, smem_u32(&sm.q[0]) + kTileBytes, bar, entry_of(rd.item[1] - bh1 * Tb), bh1);
                }
                __syncwarp();
                ++nq;
                return true;
            };
            if (is_k && steps == 0 && !load_q()) dead = true;
            for (int t0 = 0; t0 < steps && !dead; t0 += 32) {
                uint32_t ent[2] = {0u, 0u};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int t = t0 + lane, i = rd.tb[h] + t - p.ntxt;  // entry of the item's list
                    if (t < rd.nb[h] && i >= 0)
                        ent[h] = entry_of(p.idx ? clamp_label(ld_list<kSel>(p.idx + (size_t)rd.item[h] * p.keep + i), Tb) : i);
                }
                const int te = min(t0 + 32, steps);
                for (int t = t0; t < te; ++t) {
                    const uint32_t st = g % kStages, full = full0 + 8 * st, dst = tile0 + st * kPairBytes;
                    const uint32_t e0 = __shfl_sync(0xffffffffu, ent[0], t - t0);
                    const uint32_t e1 = __shfl_sync(0xffffffffu, ent[1], t - t0);
                    const bool ok = mbar_wait(empty0 + 8 * st, ((g / kStages) & 1) ^ 1, abortf, p.budget_ns);
                    if (!__all_sync(0xffffffffu, ok)) {
                        dead = true;
                        break;
                    }
                    if (elect_one_sync()) {
                        const bool a = t < rd.nb[0], b = t < rd.nb[1];
                        mbar_arrive_expect_tx(full, (a + b) * kTileBytes);
                        if (!(hold && g == 0)) {
                            // text keys / values [64 pos, 64 pos + 64) at positions pos < ntxt, zero past T_txt
                            if (a) {
                                if (rd.tb[0] + t < p.ntxt) tma_load_3d(dst, mt, full, 0, (rd.tb[0] + t) * 64, bh0);
                                else window_boxes_e(m4, dst, full, e0, bh0);
                            }
                            if (b) {
                                if (rd.tb[1] + t < p.ntxt)
                                    tma_load_3d(dst + kTileBytes, mt, full, 0, (rd.tb[1] + t) * 64, bh1);
                                else
                                    window_boxes_e(m4, dst + kTileBytes, full, e1, bh1);
                            }
                        }
                        TL_TILE(slot, g, is_k ? tl::kKIssue : tl::kVIssue);
                    }
                    __syncwarp();
                    ++g;
                    // the round's Q after its first K: it waits longest
                    if (is_k && t == 0 && !load_q()) {
                        dead = true;
                        break;
                    }
                }
            }
        }
    } else if (role == kQK) {
        // ------------------------------------------------------------ QK issuer
        // S_g = [Q_A; Q_B] [K_A; K_B]^T once the softmax holds S_{g-1} in registers (N=64 on the one
        // half's keys where only one takes part). MMAs and commits are issued under an elect.sync
        // taken at the issue site: the compiler then keeps the descriptors on the uniform datapath
        // (measured: 4 MMAs + commit issue in about 280 cycles, against about 480 under a
        // precomputed lane test). elect.sync picks the same lane of a full warp every time, so a
        // commit always follows the MMAs of its own thread.
        const uint32_t kbase = smem_u32(&sm.k[0][0]);
        for (int r = 0; r < rounds && !*abortf; ++r) {
            const Round rd = get_round<kSel>(p, ct, r);
            const int steps = max(rd.nb[0], rd.nb[1]), both = min(rd.nb[0], rd.nb[1]);
            const uint32_t one_b = rd.nb[1] > rd.nb[0] ? 1u : 0u;  // the half of the steps past `both`
            const uint32_t qaddr = smem_u32(&sm.q[0]);
            wait_phase(smem_u32(&ct.q_full), r & 1, abort_at, p.budget_ns);
            if (steps == 0 && elect_one_sync()) mma_commit(smem_u32(&ct.q_empty));
            for (int t = 0; t < steps; ++t, ++g) {
                const uint32_t st = g % kStages;
                wait_phase(smem_u32(&ct.k_full[st]), (g / kStages) & 1, abort_at, p.budget_ns);
                // QK_g follows PV_{g-2}: the softmax, which sees S_g, then knows its P buffer is free (a wait of
                // its own there cost 7 % of the whole kernel)
                if (g >= 2) wait_phase(smem_u32(&ct.o_full[g & 1]), ((g >> 1) - 1) & 1, abort_at, p.budget_ns);
                if (g >= 1) wait_phase(smem_u32(&ct.s_free), (g - 1) & 1, abort_at, p.budget_ns);
                if (lane == 0) TL_TILE(slot, g, tl::kSFree);
                tc_fence_after();
                if (elect_one_sync()) {
                    const uint32_t off = t < both ? 0u : one_b;
                    const uint32_t idesc = t < both ? kIdescQK : kIdescQK1;
                    const uint64_t adesc = sdesc_sw128(qaddr, 16, 1024);
                    const uint64_t bdesc = sdesc_sw128(kbase + st * kPairBytes + off * kTileBytes, 16, 1024);
                    const uint32_t d = tbase + kColS + off * 64;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        mma_ss(d, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc, k > 0 ? 1u : 0u);
                    mma_commit(smem_u32(&ct.s_full));
                    mma_commit(smem_u32(&ct.k_empty[st]));
                    if (t == steps - 1) mma_commit(smem_u32(&ct.q_empty));  // last read of this Q pair
                    TL_TILE(slot, g, tl::kQKIssue);
                }
                __syncwarp();
            }
        }
        dead = *abortf != 0;
    } else if (role == kPV) {
        // ------------------------------------------------------------ PV issuer
        // O_h += P_h V_h of both halves once the softmax has stored P_g and V_g has landed; all PVs
        // of a pipeline are issued by this one thread, so they accumulate into O in order. (One
        // issuer for QK and PV took 2000 cycles a step: its waits and issues do not overlap.)
        const uint32_t vbase = smem_u32(&sm.v[0][0]);
        for (int r = 0; r < rounds && !*abortf; ++r) {
            const Round rd = get_round<kSel>(p, ct, r);
            const int steps = max(rd.nb[0], rd.nb[1]);
            for (int t = 0; t < steps; ++t, ++g) {
                const uint32_t pb = g & 1, st = g % kStages;
                wait_phase(smem_u32(&ct.v_full[st]), (g / kStages) & 1, abort_at, p.budget_ns);
                wait_phase(smem_u32(&ct.p_full[pb]), (g >> 1) & 1, abort_at, p.budget_ns);
                if (lane == 0) TL_TILE(slot, g, tl::kPVReady);
                tc_fence_after();
                if (elect_one_sync()) {
                    const uint32_t pcol = tbase + kColP + pb * 32;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (t >= rd.nb[h]) continue;
                        const uint64_t vdesc = sdesc_sw128(vbase + st * kPairBytes + h * kTileBytes, 8192, 1024);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            mma_ts_half(h, tbase + kColO, pcol + k * 8, vdesc + (uint64_t)(k * 128), kIdescPV,
                                        (t > 0 || k > 0) ? 1u : 0u);
                    }
                    mma_commit(smem_u32(&ct.o_full[pb]));
                    mma_commit(smem_u32(&ct.v_empty[st]));
                    TL_TILE(slot, g, tl::kPVIssue);
                }
                __syncwarp();
            }
        }
        dead = *abortf != 0;
    } else if (role == kSoftmax) {
        // ------------------------------------------------------------ softmax and output
        const int quad = gwarp & 3;  // TMEM lane quadrant of this warp
        const int half = quad >> 1;
        const int row = (quad & 1) * 32 + lane;  // tile row of the half's item
        const uint32_t tq = tbase + (static_cast<uint32_t>(quad * 32) << 16);
        const uint32_t scol = tq + kColS + half * 64, ocol = tq + kColO;
        const float c = p.scale_log2;
        // The last round's item, whose O is written after this round's first exps: its row statistics
        // stay here; its last PV is that of step g - 1.
        bool owed = false;
        float done_m = 0.f, done_l = 0.f;
        auto wait_pv = [&](uint32_t x) {  // PV_x has finished
            wait_phase(smem_u32(&ct.o_full[x & 1]), (x >> 1) & 1, abort_at, p.budget_ns);
            tc_fence_after();
        };
        // writes the rows of round r's item, whose last PV is that of step `last`
        auto finish = [&](uint32_t last, int r) {
            if (quad == 0 && lane == 0) TL_ITEM(slot, (uint32_t)r, tl::kEpiStart);
            wait_pv(last);
            if (quad == 0 && lane == 0) TL_ITEM(slot, (uint32_t)r, tl::kEpiO);
            const Round rd = get_round<kSel>(p, ct, r);
            store_row(p, half ? rd.item[1] : rd.item[0], row, ocol, done_m, done_l);
            if (quad == 0 && lane == 0) TL_ITEM(slot, (uint32_t)r, tl::kEpiDone);
            tc_fence_before();
            owed = false;
        };
        bool split = false;
        for (int r = 0; r < rounds && !*abortf; ++r) {
            int nb, steps, mask_t;  // mask_t: the step of the last text block, if that one is ragged
            bool parted;            // half B has blocks (of a split item: there is something to merge)
            {
                const Round rd = get_round<kSel>(p, ct, r);
                nb = half ? rd.nb[1] : rd.nb[0];
                steps = max(rd.nb[0], rd.nb[1]);
                mask_t = (p.t_txt & 63) ? p.ntxt - 1 - (half ? rd.tb[1] : rd.tb[0]) : -1;
                split = rd.split;
                parted = rd.nb[1] > 0;
                if (steps == 0) {  // empty lists: nothing was multiplied; O = 0, lse = -inf
                    if (owed) finish(g - 1, r - 1);
                    if (!split || half == 0)
                        store_row(p, half ? rd.item[1] : rd.item[0], row, ocol, 0.f, 0.f);
                    split = false;
                    continue;
                }
            }
            float m_used = 0.f, l = 0.f;
            for (int t = 0; t < nb; ++t, ++g) {
                wait_phase(smem_u32(&ct.s_full), g & 1, abort_at, p.budget_ns);
                if (quad == 0 && lane == 0) TL_TILE(slot, g, tl::kSmxStart);
                tc_fence_after();
                uint32_t sr[64];
                tmem_ld_32x32b_x32(scol, &sr[0]);
                tmem_ld_32x32b_x32(scol + 32, &sr[32]);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ct.s_free));
                if (quad == 0 && lane == 0) TL_TILE(slot, g, tl::kSLoaded);
                if (t == mask_t) {
                    // the last text block: its columns past T_txt are zero-filled keys, not keys
#pragma unroll
                    for (int i = 0; i < 64; ++i)
                        if (i >= (p.t_txt & 63)) sr[i] = __float_as_uint(-INFINITY);
                }
                const float2 c2 = make_float2(c, c);
                // P = exp2(s c - m) in bf16 to tensor memory; returns the thread's row sum of it. Packed
                // fp32x2 arithmetic (two columns per op).
                auto exps = [&]() -> float {
                    const float2 nm2 = make_float2(-m_used, -m_used);
                    float2 ls2[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f),
                                     make_float2(0.f, 0.f)};
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) {
                        uint32_t pk[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float2 x = __ffma2_rn(make_float2(__uint_as_float(sr[32 * h2 + 2 * i]),
                                                                    __uint_as_float(sr[32 * h2 + 2 * i + 1])), c2, nm2);
                            const float2 pp = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                            ls2[i & 3] = __fadd2_rn(ls2[i & 3], pp);
                            pk[i] = pack_bf16(pp.x, pp.y);
                        }
                        tmem_st_32x32b_x16(tq + kColP + (g & 1) * 32 + h2 * 16, pk);
                    }
                    const float2 lsum = __fadd2_rn(__fadd2_rn(ls2[0], ls2[1]), __fadd2_rn(ls2[2], ls2[3]));
                    return lsum.x + lsum.y;
                };
                // the first step only takes its maximum; later ones nearly always skip it (141 of 536
                // cycles of a warp's step, two warps a scheduler)
                float ls = t == 0 ? INFINITY : exps();
                const bool over = !(ls <= kRaise);
                if (__any_sync(0xffffffffu, over)) {
                    float mx;
                    {
                        float t8[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) t8[i] = __uint_as_float(sr[i]);
#pragma unroll
                        for (int j = 8; j < 56; j += 16)
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                t8[i] = max3(t8[i], __uint_as_float(sr[j + i]), __uint_as_float(sr[j + 8 + i]));
#pragma unroll
                        for (int i = 0; i < 8; ++i) t8[i] = fmaxf(t8[i], __uint_as_float(sr[56 + i]));
                        mx = fmaxf(max3(max3(t8[0], t8[1], t8[2]), t8[3], t8[4]), max3(t8[5], t8[6], t8[7]));
                    }
                    const float mx2 = fmaxf(mx * c, -3.0e38f);  // finite, so that scores of -inf give P = 0
                    const float alpha = over && t > 0 ? fast_exp2(m_used - mx2) : 1.f;
                    m_used = over ? mx2 : m_used;
                    l *= alpha;
                    if (t > 0) {
                        wait_pv(g - 1);
#pragma unroll
                        for (int h2 = 0; h2 < 4; ++h2) {
                            uint32_t o[16];
                            tmem_ld_32x32b_x16(ocol + h2 * 16, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tmem_st_32x32b_x16(ocol + h2 * 16, o);
                        }
                    }
                    ls = exps();
                }
                l += ls;
                if (quad == 0 && lane == 0) TL_TILE(slot, g, tl::kSmxExp);
                if (t == 0 && owed) finish(g - 1, r - 1);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ct.p_full[g & 1]));
                if (quad == 0 && lane == 0) TL_TILE(slot, g, tl::kPStored);
            }
            // steps that only the other half takes part in
            for (int t = nb; t < steps; ++t, ++g) {
                wait_phase(smem_u32(&ct.s_full), g & 1, abort_at, p.budget_ns);
                if (t == 0 && owed) finish(g - 1, r - 1);
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(smem_u32(&ct.s_free));
                    mbar_arrive(smem_u32(&ct.p_full[g & 1]));
                }
            }
            if (split && !parted) {  // one block: half A has all of it
                split = false;
                if (half) break;
            }
            owed = true;
            done_m = m_used;
            done_l = l;
        }
        // the pipeline's last item or items
        if (owed && !split) finish(g - 1, rounds - 1);
        if (split) {
            // a split item: half B leaves its part in the K ring (no copy or product uses it any
            // more), half A adds it to its own (two partial softmax sums) and writes the rows
            float* part = reinterpret_cast<float*>(&sm.k[0][0]) + row * kD;
            float2* stat = reinterpret_cast<float2*>(&sm.k[1][0]) + row;
            wait_pv(g - 1);
            if (half == 1) {
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    uint32_t o[32];
                    tmem_ld_32x32b_x32(ocol + h2 * 32, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *reinterpret_cast<float4*>(part + 4 * ((8 * h2 + i) ^ (row & 15))) =
                            make_float4(__uint_as_float(o[4 * i]), __uint_as_float(o[4 * i + 1]),
                                        __uint_as_float(o[4 * i + 2]), __uint_as_float(o[4 * i + 3]));
                }
                *stat = make_float2(done_m, done_l);
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ct.merged));
            } else {
                wait_phase(smem_u32(&ct.merged), 0, abort_at, p.budget_ns);
                const float2 os = *stat;
                const bool a_ok = done_l != 0.f, b_ok = os.y != 0.f;
                const float m = a_ok ? (b_ok ? fmaxf(done_m, os.x) : done_m) : os.x;
                const float wa = a_ok ? fast_exp2(done_m - m) : 0.f, wb = b_ok ? fast_exp2(os.x - m) : 0.f;
                store_row(p, ct.last, row, ocol, m, (a_ok ? done_l * wa : 0.f) + (b_ok ? os.y * wb : 0.f), part, wa,
                          wb, a_ok, b_ok);
            }
            tc_fence_before();
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
    if (soft && threadIdx.x % (kSoftWarps * 32) == 0) TL_CTA(slot == 0 ? tl::kSlot0End : tl::kSlot1End);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (gwarp == 1) tmem_dealloc(cs.tmem_base, kTmemCols);
    if (threadIdx.x == 0) TL_CTA(tl::kEnd);
}

// [B*heads][T][d] bf16 as a 3-D map with 64-row boxes (128-byte swizzle); rows past T read
// as zeros.
bool encode_rows_map(CUtensorMap* m, const void* base, int BH, int T)
{
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)kD, (cuuint64_t)T, (cuuint64_t)BH};
    cuuint64_t strides[2] = {(cuuint64_t)kD * 2, (cuuint64_t)T * kD * 2};
    cuuint32_t box[3] = {kD, 64, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int num_sms() { return device_sm_count(); }
PerDeviceOnce g_attn_attr;  // the kernel's shared-memory attributes, set once per device

}  // namespace

namespace {
// Items per SM up to which the selection (and the pooling) run inside the attention launch. A CTA has
// 16 warps, one item each; beyond that its rows queue up while the tensor pipe waits, and separate
// launches, which give every SM several CTAs' warps, are faster: 2048 px (40 items) 395 -> 360 us a
// layer, four 1024 px images (40) 187 -> 176; at one 1024 px image (10) the single launch is (48.2
// against 49.3 us). ssba_build_mask and ssba_forward are two launches (the mask kernel, which pools without a
// grid barrier but does not write the means that these calls return): 24 heads, one launch and those two,
// 256 px 12.0, 9.2 us, 512 px 16.0, 14.4, 1024 px 47.0, 46.9.
constexpr int kSelItems = 16;
int max_grid() { return num_sms(); }
size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }
}  // namespace

// Bytes of the forward workspace. Only its last 256 are used, by the grid barrier of the launch that
// pools; the rest is the size callers have always had to bring (a split schedule's counters, row
// statistics and partial O, two pipelines an SM), so that what was too small stays too small.
size_t attn_tc_workspace_bytes()
{
    const size_t boundaries = (size_t)kSlots * max_grid() + 1;
    return align256(boundaries * 4 * sizeof(int)) + align256(boundaries * 2 * kRows * sizeof(float2)) +
           align256(boundaries * 2 * kRows * kD * sizeof(float)) + 256;
}

int launch_attn_tc_bf16(const ssba_desc& d, const Grid& g, int keep, float scale, const void* Q, const void* K,
                        const void* V, const int32_t* idx, const int32_t* cnt, void* O, float* lse, void* ws,
                        size_t ws_bytes, cudaStream_t st, uint64_t budget_ns, int withhold, const void* Kt,
                        const void* Vt, int t_txt, const float* sel_qb, const float* sel_kb, float* sel_scores,
                        bool pool)
{
    if (pool && (!ws || !sel_qb || !sel_kb)) {
        set_error("ssba_forward_fused: needs a forward workspace and the block-mean buffers");
        return SSBA_ERR_WORKSPACE;
    }
    if (sel_qb && (g.Tb() > kWinCap || t_txt > 0 || !idx || !cnt)) {
        set_error("ssba_forward_select: needs Tb <= 256, no text segment and list outputs");
        return SSBA_ERR_UNSUPPORTED;
    }
    if (d.head_dim != kD || g.blk != 8 || (g.sr % 4) || (g.sc % 4)) {
        set_error("ssba_forward (bf16): needs head_dim=64, block=8 and shifts that are multiples of 4");
        return SSBA_ERR_UNSUPPORTED;
    }
    if (g.H >= 32768 || g.W >= 32768) {
        set_error("ssba_forward (bf16): H_tok and W_tok must be below 32768");
        return SSBA_ERR_UNSUPPORTED;
    }
    if (ws && ws_bytes < attn_tc_workspace_bytes()) {
        set_error("ssba_forward (bf16): workspace of %zu bytes, %zu needed", ws_bytes, attn_tc_workspace_bytes());
        return SSBA_ERR_WORKSPACE;
    }
    const int BH = d.B * d.heads;
    if (sel_qb && withhold == 0 && BH * g.Tb() > kSelItems * max_grid()) {
        int rc = pool ? launch_pool_blocks(d, g, Q, K, const_cast<float*>(sel_qb), const_cast<float*>(sel_kb), st)
                      : SSBA_OK;
        if (rc == SSBA_OK)
            rc = launch_select(d, g, keep, sel_qb, sel_kb, const_cast<int32_t*>(idx), const_cast<int32_t*>(cnt),
                               sel_scores, st);
        if (rc != SSBA_OK) return rc;
        return launch_attn_tc_bf16(d, g, keep, scale, Q, K, V, idx, cnt, O, lse, ws, ws_bytes, st, budget_ns);
    }
    TileMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (!encode_window_maps(maps.q, Q, BH, g.H, g.W) || !encode_window_maps(maps.k, K, BH, g.H, g.W) ||
        !encode_window_maps(maps.v, V, BH, g.H, g.W)) {
        set_error("ssba_forward (bf16): cuTensorMapEncodeTiled failed");
        return SSBA_ERR_CUDA;
    }
    if (t_txt > 0 && (!encode_rows_map(&maps.kt, Kt, BH, t_txt) || !encode_rows_map(&maps.vt, Vt, BH, t_txt))) {
        set_error("ssba_forward_joint: cuTensorMapEncodeTiled failed for the text keys/values");
        return SSBA_ERR_CUDA;
    }
    TcParams p;
    p.O = static_cast<__nv_bfloat16*>(O);
    p.lse = lse;
    p.idx = idx;
    p.cnt = cnt;
    p.g = g;
    p.keep = keep;
    p.t_txt = t_txt > 0 ? t_txt : 0;
    p.ntxt = (p.t_txt + 63) / 64;
    p.units = p.ntxt + keep;
    p.num_items = BH * g.Tb();
    p.scale_log2 = scale * 1.4426950408889634f;
    p.budget_ns = budget_ns;
    p.withhold = withhold;
    p.sel_qb = sel_qb;
    p.sel_kb = sel_kb;
    p.sel_cnt = const_cast<int32_t*>(cnt);
    p.sel_scores = sel_scores;
    p.pool_q = pool ? static_cast<const __nv_bfloat16*>(Q) : nullptr;
    p.pool_k = pool ? static_cast<const __nv_bfloat16*>(K) : nullptr;
    p.gsync = pool ? reinterpret_cast<unsigned*>(static_cast<char*>(ws) + attn_tc_workspace_bytes() - 256) : nullptr;
    p.status = device_status_word();
    if (!p.status) {
        set_error("ssba_forward (bf16): could not resolve the device status word");
        return SSBA_ERR_CUDA;
    }
    const size_t smem = sizeof(SmemLayout) + 1024;
    g_attn_attr.run([smem] {
        for (auto k : {ssba_attn_tc_kernel<false>, ssba_attn_tc_kernel<true>}) {
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        }
    });
    // One CTA fits an SM (shared memory), so each CTA runs kSlots pipelines; the persistent
    // grid has one CTA per SM, fewer for small problems (one item a pipeline: with one a CTA the next
    // layer's mask finds too few free SMs to start early, 13.0 against 10.0 us a 256 px layer).
    const int want = (p.num_items + kSlots - 1) / kSlots;
    const int grid = want < max_grid() ? want : max_grid();
    // programmatic dependent launch: the kernel may start (barriers, tensor memory, window
    // table) while the previous grid on the stream finishes; it waits for that grid before
    // reading any input
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, sel_qb ? ssba_attn_tc_kernel<true> : ssba_attn_tc_kernel<false>, maps, p);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("ssba_attn_tc_kernel launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

// Timeline of the last launch of the attention kernel on the current device (timeline build only).
int timeline_read(unsigned long long* cta, unsigned* tile, unsigned* item)
{
#ifdef SSBA_TIMELINE
    if (cudaMemcpyFromSymbol(cta, tl::cta_ev, sizeof(tl::cta_ev)) != cudaSuccess ||
        cudaMemcpyFromSymbol(tile, tl::tile_ev, sizeof(tl::tile_ev)) != cudaSuccess ||
        cudaMemcpyFromSymbol(item, tl::item_ev, sizeof(tl::item_ev)) != cudaSuccess) {
        set_error("ssba_timeline_read: copy from the device failed");
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
#else
    (void)cta;
    (void)tile;
    (void)item;
    set_error("ssba_timeline_read: this library was built without -DSSBA_TIMELINE");
    return SSBA_ERR_UNSUPPORTED;
#endif
}

// Dense attention: the 128-token-tile kernel (attn_dense.cu) when N is a multiple of 128, else
// this kernel with no list, every key block visited in label order with query tiles of one 8x8
// block each (unshifted grid).
int launch_dense_tc_bf16(const ssba_desc& d, float scale, const void* Q, const void* K, const void* V, void* O,
                         float* lse, void* ws, size_t ws_bytes, cudaStream_t st)
{
    if (ws && ws_bytes < attn_tc_workspace_bytes()) {  // the rules of ssba_forward, whichever kernel runs
        set_error("ssba_forward_dense: workspace of %zu bytes, %zu needed", ws_bytes, attn_tc_workspace_bytes());
        return SSBA_ERR_WORKSPACE;
    }
    const int rc = launch_dense_m128(d, scale, Q, K, V, O, lse, st);
    if (rc != SSBA_ERR_UNSUPPORTED) return rc;
    if (d.head_dim != kD || d.H_tok % 8 || d.W_tok % 8) {
        set_error("ssba_forward_dense: needs head_dim=64 and H_tok, W_tok multiples of 8");
        return SSBA_ERR_UNSUPPORTED;
    }
    Grid g;
    g.H = d.H_tok;
    g.W = d.W_tok;
    g.blk = 8;
    g.sr = 0;
    g.sc = 0;
    g.bw = d.W_tok / 8;
    return launch_attn_tc_bf16(d, g, g.Tb(), scale, Q, K, V, nullptr, nullptr, O, lse, ws, ws_bytes, st);
}

}  // namespace ssba
