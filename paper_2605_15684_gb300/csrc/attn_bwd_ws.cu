// attn_bwd_ws.cu -- the tensor-core backward (gradients of Algorithm 1's SparseAttention over
// the kept blocks; the chain rule, the paper gives no backward) as one persistent,
// warp-specialised launch, for shifts that are multiples of 4, so that every window is one,
// two or four TMA boxes (window.cuh). The products, operand layouts and per-pair arithmetic are
// those of attn_bwd_tc.cu; what changes is who waits on what.
//
// Work items: a key block's dK, dV or a query block's dQ, of one (batch, head). The first item
// of a CTA is its index; the others come from a counter in the workspace that the row kernel
// zeroes. Key-block items come first (their lengths vary), query-block items fill in behind.
//   warp 11    producer: publishes each item (role, head, block, count and its list of other
//              blocks: the forward's list for dQ, the transposed list the row kernel built for
//              dK, dV) in one of two item slots; copies the item's resident tiles by TMA (two
//              buffers, by item parity) and each pair's streamed tiles (a ring of three), each
//              with the 512-byte row of its block's statistics (lse, D) that the compute warps
//              use (the row kernel writes them by block, in tile order: one bulk copy).
//   warps 8-10 lane 0 of each issues a share of the MMAs: warp 8 S, warp 9 dP, into the same
//              TMEM columns once the compute warps hold the last pair's in registers; warp 10 the
//              accumulating products of a pair, once its bf16 operands are stored. (Four products
//              take a thread about 450 cycles to issue. With dK on S's thread and dV on dP's, a
//              pair's S waited 860 cycles for its thread.)
//   warps 0-7  the exps and the bf16 operands of each pair, two warps per TMEM lane quadrant
//              (16 of a row's 64 columns a thread), and each item's epilogue (the accumulators
//              to global memory, fp32).
// Pairs are counted across items: the next item's tiles arrive while the last item computes,
// and its first products run while the compute warps store the last item's gradients.
// What bounds it: the tensor pipe's 64 x 64 products and the chain of hand-offs between them (S, dP ->
// registers -> bf16 operands -> products). At 2048 px a pair takes a CTA 1810 cycles, of which the products
// of the SM's two CTAs take about 1230 (44 cycles each, 14 a pair); alone on its SM a CTA takes 1540. So
// the compute warps' instructions count: the statistics come as addends for packed two-column
// arithmetic, and the pair loop's waits return no verdict (wait_phase). 24 heads, a call, before these
// and now: 1024 px 139.4, 132.2 us, four 1024 px images 701, 664, 2048 px 1556, 1460 (the threads that
// issue are 1.2 us of the first).
// Tile rows follow the TMA box order (tile_row_pos). Every wait is bounded; on a timeout the
// CTA records SSBA_ERR_TIMEOUT, waits (bounded) for its copies and MMAs in flight, and returns. (After one
// the compute warps may run on, on whatever their own tiles hold, and write their items' rows: the gradients
// are undefined then. A wait that ran out is reported even where its phase completed later.)
#include <algorithm>
#include <cstdint>

#include "bwd_tile.cuh"
#include "common.cuh"
#include "ptx.cuh"
#include "window.cuh"

namespace ssba {

namespace {

using namespace ptx;
using namespace win;
using namespace bwd;

constexpr int kCompute = 256;   // warps 0-7, two per TMEM lane quadrant
constexpr int kIssuer0 = 256;   // lane 0 of warp 8: S
constexpr int kIssuer1 = 288;   // lane 0 of warp 9: dP
constexpr int kIssuer2 = 320;   // lane 0 of warp 10: the accumulating products
constexpr int kIssuers = 3;     // commit to drain
constexpr int kSdpIssuers = 2;  // commit to bar_s, ab_empty
constexpr int kProducer = 11;   // warp
constexpr int kThreads = 384;
constexpr int kRing = 3;        // streamed tile slots
constexpr int kDone = -1;       // role of the item slot that ends a CTA's work
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kColS = 0, kColDP = 64, kColA0 = 128, kColA1 = 192;
constexpr size_t kSmemBytes = 104 * 1024;  // two CTAs per SM (TMEM: 2 x 256 columns)

struct WsMaps {
    CUtensorMap q[4], k[4], v[4], o[4];  // Q, K, V, dO as window boxes (o: dO)
};

struct alignas(1024) WsSmem {
    uint8_t a[2][kTile];      // item tiles by item parity: dQ item Q_i, dK/dV item K_j
    uint8_t b[2][kTile];      //                            dO_i,         V_j
    uint8_t x[kRing][kTile];  // pair tiles: dQ item K_j, dK/dV item Q_i
    uint8_t y[kRing][kTile];  //             V_j,         dO_i
    uint8_t e[2][kTile];      // bf16 operands: dS (e[0]); P^T and dS^T
    float4 pld[kRing][kT / 2];  // dK/dV pair: the statistics of its query rows (BwdParams::ld)
    float4 ild[2][kT / 2];      // dQ item: of its rows
    int list[2][256];         // the item's other blocks, in pair order (producer only)
    uint32_t win[256];        // label -> packed window entry (window_entry)
    int4 info[2];             // role (0 dQ, 1 dK/dV, kDone), bh, label, n
    uint64_t item_full[2];    // producer lane 0, after the slot is written
    uint64_t item_empty[2];   // the 8 compute warps and the 3 issuers have read the slot
    uint64_t ab_full[2];      // TMA bytes of the item tiles (and, for dQ, of its ild row)
    uint64_t ab_empty[2];     // MMA commits (the S and dP issuers) after the item's last S, dP
    uint64_t tile_full[kRing];   // TMA bytes of a pair's tiles (and, for dK/dV, of its pld row)
    uint64_t tile_empty[kRing];  // MMA commit after the pair's accumulating products
    uint64_t bar_s;           // MMA commits (the S and dP issuers): S, dP of the pair in TMEM
    uint64_t s_free;          // 8 compute warps: S, dP in registers
    uint64_t e_full;          // 8 compute warps: the pair's bf16 operands stored
    uint64_t bar_a;           // MMA commit: the pair's accumulating products
    uint64_t drain;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(WsSmem) + 1024 <= kSmemBytes, "shared memory");

__device__ __forceinline__ WsSmem& smem_layout()
{
    extern __shared__ uint8_t raw[];
    return *reinterpret_cast<WsSmem*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~static_cast<uintptr_t>(1023));
}

// A warp's bounded wait: every lane must see the phase, so a timeout takes the warp out whole.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abortf, uint64_t budget_ns)
{
    const bool ok = mbar_wait(bar, parity, abortf, budget_ns);
    return __all_sync(0xffffffffu, ok);
}

// One arrive per warp, after every lane's earlier TMEM loads and shared-memory writes.
__device__ __forceinline__ void warp_arrive(uint32_t bar)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

// Token of tile row r of block `label` (TMA box order).
__device__ __forceinline__ int tile_token(const Grid& g, int label, int r)
{
    return g.token(label, tile_row_pos(g, label, r));
}

constexpr uint32_t kLdRow = kT * sizeof(float2);  // 512 bytes of statistics per block

// An item slot's shape, read after its mbarrier wait.
__device__ __forceinline__ int4 read_info(const int4* q)
{
    const volatile int* v = reinterpret_cast<const volatile int*>(q);
    return make_int4(v[0], v[1], v[2], v[3]);
}

// Item w: [0, nk) key blocks (role 1), then query blocks (role 0), bh-major.
__device__ __forceinline__ int4 decode_item(int w, int nk, int Tb)
{
    const bool key = w < nk;
    const int u = key ? w : w - nk, bh = u / Tb;
    return make_int4(key ? 1 : 0, bh, u - bh * Tb, 0);
}

// Warp 11. nk = number of key-block items (B * heads * Tb), total = 2 nk. Returns false on a
// timeout. P counts the pairs whose tiles were issued, kab the items whose tiles were issued
// (after a timeout the teardown waits for the last copies of each barrier).
__device__ bool produce(const WsMaps& maps, const BwdParams& p, WsSmem& sm, const int nk, uint32_t& P, int& kab)
{
    const int lane = threadIdx.x & 31;
    const Grid& g = p.g;
    const int Tb = g.Tb();
    volatile int* abortf = &sm.abort_flag;
    grid_dep_wait();  // D, the counter and the transposed lists come from the row kernel
    int w = blockIdx.x;
    kab = 0;
    for (int k = 0;; ++k) {
        const int s = k & 1;
        if (k >= 2 && !warp_wait(smem_u32(&sm.item_empty[s]), ((k >> 1) + 1) & 1, abortf, p.budget_ns))
            return false;
        if (w >= 2 * nk) {  // no work left: the end marker
            if (lane == 0) {
                sm.info[s] = make_int4(kDone, 0, 0, 0);
                mbar_arrive(smem_u32(&sm.item_full[s]));
            }
            return true;
        }
        const int4 it = decode_item(w, nk, Tb);
        const int role = it.x, bh = it.y, label = it.z;
        const size_t brow = (size_t)bh * Tb + label;
        int n;
        const int32_t* src;
        if (role == 1) {  // dK, dV: the query blocks whose lists hold this key block, ascending
            n = min(max(__ldg(p.tcnt + brow), 0), Tb);
            src = p.tlist + __ldg(p.toff + brow);
        } else {  // dQ: the forward's list
            n = min(max(__ldg(p.cnt + brow), 0), p.keep);
            src = p.idx + brow * p.keep;
        }
        for (int i = lane; i < n; i += 32) sm.list[s][i] = min(max(__ldg(src + i), 0), Tb - 1);
        __syncwarp();
        if (lane == 0) {
            sm.info[s] = make_int4(role, bh, label, n);
            mbar_arrive(smem_u32(&sm.item_full[s]));
        }
        // the item's resident tiles, once the item two back has issued its last S, dP
        if (k >= 2 && !warp_wait(smem_u32(&sm.ab_empty[s]), ((k >> 1) + 1) & 1, abortf, p.budget_ns)) return false;
        if (lane == 0) {
            const uint32_t bar = smem_u32(&sm.ab_full[s]), e = sm.win[label];
            mbar_arrive_expect_tx(bar, 2 * kTile + (role ? 0 : kLdRow));
            window_boxes_e(role ? maps.k : maps.q, smem_u32(sm.a[s]), bar, e, bh);
            window_boxes_e(role ? maps.v : maps.o, smem_u32(sm.b[s]), bar, e, bh);
            if (!role) bulk_load(smem_u32(sm.ild[s]), p.ld + brow * (kT / 2), kLdRow, bar);
        }
        ++kab;
        // the pairs' streamed tiles, each once the pair three back has finished its products
        for (int t = 0; t < n; ++t, ++P) {
            const int r = (int)(P % kRing);
            if (P >= kRing && !warp_wait(smem_u32(&sm.tile_empty[r]), ((P / kRing) + 1) & 1, abortf, p.budget_ns))
                return false;
            const int j = sm.list[s][t];
            // test hook: CTA 0 announces its first pair's bytes and copies nothing, so that the
            // waits on them run out
            const bool hold = p.withhold == 1 && P == 0 && blockIdx.x == 0;
            if (lane == 0) {
                const uint32_t bar = smem_u32(&sm.tile_full[r]), e = sm.win[j];
                mbar_arrive_expect_tx(bar, 2 * kTile + (role ? kLdRow : 0));
                if (!hold) {
                    window_boxes_e(role ? maps.q : maps.k, smem_u32(sm.x[r]), bar, e, bh);
                    window_boxes_e(role ? maps.o : maps.v, smem_u32(sm.y[r]), bar, e, bh);
                    if (role) bulk_load(smem_u32(sm.pld[r]), p.ld + ((size_t)bh * Tb + j) * (kT / 2), kLdRow, bar);
                }
            }
        }
        int next = 0;
        if (lane == 0) next = (int)gridDim.x + atomicAdd(p.ctr, 1);
        w = __shfl_sync(0xffffffffu, next, 0);
    }
}

// Lane 0 of warp 10: every pair's accumulating products, in pair order, once its bf16 operands are stored:
// dQ += dS K of a query-block pair, dV += P^T dO and dK += dS^T Q of a key-block pair. (A pair's operands
// are made from its S and dP, so those are done with the tiles by then: the commits here are all that
// bar_a and tile_empty count.) Returns false on a timeout.
__device__ bool issue_acc(const BwdParams& p, WsSmem& sm)
{
    volatile int* abortf = &sm.abort_flag;
    const uint32_t tb0 = sm.tmem_base;
    uint32_t P = 0;
    for (int k = 0;; ++k) {
        const int s = k & 1;
        if (!mbar_wait(smem_u32(&sm.item_full[s]), (k >> 1) & 1, abortf, p.budget_ns)) return false;
        const int4 inf = read_info(&sm.info[s]);
        mbar_arrive(smem_u32(&sm.item_empty[s]));
        if (inf.x == kDone) return true;
        const int role = inf.x, n = inf.w;
        for (int t = 0; t < n; ++t, ++P) {
            const int r = (int)(P % kRing);
            if (!mbar_wait(smem_u32(&sm.tile_full[r]), (P / kRing) & 1, abortf, p.budget_ns)) return false;
            if (!mbar_wait(smem_u32(&sm.e_full), P & 1, abortf, p.budget_ns)) return false;
            tc_fence_after();
            if (role == 0) {
                mma_sb(tb0 + kColA0, smem_u32(sm.e[0]), smem_u32(sm.x[r]), t > 0);
            } else {
                mma_sb(tb0 + kColA0, smem_u32(sm.e[0]), smem_u32(sm.y[r]), t > 0);
                mma_sb(tb0 + kColA1, smem_u32(sm.e[1]), smem_u32(sm.x[r]), t > 0);
            }
            mma_commit(smem_u32(&sm.bar_a));
            mma_commit(smem_u32(&sm.tile_empty[r]));
        }
    }
}

// Lane 0 of warp 8 (which = 0) or 9 (which = 1): S or dP of every pair, as soon as the compute warps hold
// the last pair's in registers. Returns false on a timeout.
__device__ bool issue_sdp(const BwdParams& p, WsSmem& sm, const int which)
{
    volatile int* abortf = &sm.abort_flag;
    const uint32_t tb0 = sm.tmem_base;
    uint32_t P = 0;  // pairs issued
    for (int k = 0;; ++k) {
        const int s = k & 1;
        if (!mbar_wait(smem_u32(&sm.item_full[s]), (k >> 1) & 1, abortf, p.budget_ns)) return false;
        const int4 inf = read_info(&sm.info[s]);
        mbar_arrive(smem_u32(&sm.item_empty[s]));
        if (inf.x == kDone) return true;
        const int n = inf.w;
        if (!mbar_wait(smem_u32(&sm.ab_full[s]), (k >> 1) & 1, abortf, p.budget_ns)) return false;
        const uint32_t ab = smem_u32(which ? sm.b[s] : sm.a[s]);
        for (int t = 0; t < n; ++t, ++P) {
            const int r = (int)(P % kRing);
            if (!mbar_wait(smem_u32(&sm.tile_full[r]), (P / kRing) & 1, abortf, p.budget_ns)) return false;
            if (P > 0) wait_phase(smem_u32(&sm.s_free), (P - 1) & 1, smem_u32(&sm.abort_flag), p.budget_ns);
            tc_fence_after();
            if (which == 0)
                mma_kk(tb0 + kColS, ab, smem_u32(sm.x[r]));  // S = Q K^T (dK/dV item: S^T = K Q^T)
            else
                mma_kk(tb0 + kColDP, ab, smem_u32(sm.y[r]));  // dP = dO V^T (dP^T = V dO^T)
            mma_commit(smem_u32(&sm.bar_s));
            if (t == n - 1) mma_commit(smem_u32(&sm.ab_empty[s]));
        }
        if (n == 0) mma_commit(smem_u32(&sm.ab_empty[s]));
    }
}

// Columns [col0, col0 + 16) of this thread's row of the fp32 accumulator whose 16-column
// group starts at TMEM address taddr, times mul, to row `token` of out (one [N][64] head).
__device__ __forceinline__ void store_cols(uint32_t taddr, float* out, int token, int col0, float mul)
{
    uint32_t v[16];
    tmem_ld_16x32bx2_x16_off32(taddr, v);
    tmem_wait_ld();
    float4* dst = reinterpret_cast<float4*>(out + (size_t)token * kD + col0);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        dst[i] = make_float4(__uint_as_float(v[4 * i]) * mul, __uint_as_float(v[4 * i + 1]) * mul,
                             __uint_as_float(v[4 * i + 2]) * mul, __uint_as_float(v[4 * i + 3]) * mul);
}

// Sixteen bf16 values (8 packed pairs) of row r, 16-byte chunks c0 and c0 + 1, into the
// 128-byte-swizzled K-major tile at dst.
__device__ __forceinline__ void store_cols_bf16(uint8_t* dst, int r, int c0, const uint32_t (&v)[8])
{
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int c = c0 + i;
        *reinterpret_cast<uint4*>(dst + r * 128 + ((c ^ (r & 7)) << 4)) =
            make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
}

// Warps 0-7: warp w reads TMEM lane quadrant w % 4; thread (w, lane) owns row
// r = 16 (w % 4) + lane % 16 of the M=64 data path and its columns [col0, col0 + 16),
// col0 = 32 (lane / 16) + 16 (w / 4): two warps share each quadrant's exps. Returns false on a
// timeout.
__device__ bool compute(const BwdParams& p, WsSmem& sm)
{
    volatile int* abortf = &sm.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = warp & 3, col0 = 32 * (lane >> 4) + 16 * (warp >> 2);
    const int r = q * 16 + (lane & 15);
    // lanes 16-31 of a 16x32bx2 load read 32 columns further on: one address serves the warp
    const uint32_t tb = sm.tmem_base + (static_cast<uint32_t>(q * 32) << 16) + 16 * (warp >> 2);
    const Grid& g = p.g;
    const int N = g.H * g.W;
    const float2 c2 = make_float2(p.scale * kLog2e, p.scale * kLog2e);
    uint32_t P = 0;  // pairs done
    for (int k = 0;; ++k) {
        const int s = k & 1;
        if (!warp_wait(smem_u32(&sm.item_full[s]), (k >> 1) & 1, abortf, p.budget_ns)) return false;
        const int4 inf = read_info(&sm.info[s]);
        float2 nl2 = make_float2(0.f, 0.f), nd2 = nl2;  // -lse log2(e) and -D, twice
        if (inf.x == 0) {  // the row's statistics came with the item's tiles
            if (!warp_wait(smem_u32(&sm.ab_full[s]), (k >> 1) & 1, abortf, p.budget_ns)) return false;
            const float* st = reinterpret_cast<const float*>(&sm.ild[s][r >> 1]) + (r & 1);
            nl2 = make_float2(st[0], st[0]);
            nd2 = make_float2(st[2], st[2]);
        }
        warp_arrive(smem_u32(&sm.item_empty[s]));
        if (inf.x == kDone) return *abortf == 0;
        const int role = inf.x, bh = inf.y, label = inf.z, n = inf.w;
        for (int t = 0; t < n; ++t, ++P) {
            const int slot = (int)(P % kRing);
            wait_phase(smem_u32(&sm.bar_s), P & 1, smem_u32(&sm.abort_flag), p.budget_ns);
            tc_fence_after();
            uint32_t sv[16], dp[16];
            tmem_ld_16x32bx2_x16_off32(tb + kColS, sv);
            tmem_ld_16x32bx2_x16_off32(tb + kColDP, dp);
            tmem_wait_ld();
            tc_fence_before();
            warp_arrive(smem_u32(&sm.s_free));
            auto pair_of = [](const uint32_t (&v)[16], int i) {
                return make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            };
            auto probs = [&](const uint32_t (&v)[16], int i, float2 nl) {
                const float2 x = __ffma2_rn(pair_of(v, i), c2, nl);
                return make_float2(fast_exp2(x.x), fast_exp2(x.y));
            };
            if (role == 1) {
                // S^T, dP^T: columns are the query rows col0 + i of the pair's query block
                wait_phase(smem_u32(&sm.tile_full[slot]), (P / kRing) & 1, smem_u32(&sm.abort_flag), p.budget_ns);
                const float4* ld = sm.pld[slot] + (col0 >> 1);
                uint32_t pp[8], dd[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 qd = ld[i];  // of query rows col0 + 2 i and col0 + 2 i + 1
                    const float2 pv = probs(sv, i, make_float2(qd.x, qd.y));
                    const float2 ds = __fmul2_rn(pv, __fadd2_rn(pair_of(dp, i), make_float2(qd.z, qd.w)));
                    pp[i] = pack_bf16(pv.x, pv.y);
                    dd[i] = pack_bf16(ds.x, ds.y);
                }
                // the last pair's products have read e[] (and the tiles of its slot)
                if (P > 0) wait_phase(smem_u32(&sm.bar_a), (P - 1) & 1, smem_u32(&sm.abort_flag), p.budget_ns);
                store_cols_bf16(sm.e[0], r, col0 >> 3, pp);
                store_cols_bf16(sm.e[1], r, col0 >> 3, dd);
            } else {
                uint32_t pk[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float2 ds = __fmul2_rn(probs(sv, i, nl2), __fadd2_rn(pair_of(dp, i), nd2));
                    pk[i] = pack_bf16(ds.x, ds.y);
                }
                if (P > 0) wait_phase(smem_u32(&sm.bar_a), (P - 1) & 1, smem_u32(&sm.abort_flag), p.budget_ns);
                store_cols_bf16(sm.e[0], r, col0 >> 3, pk);
            }
            fence_proxy_async_smem();
            warp_arrive(smem_u32(&sm.e_full));
        }
        // epilogue: the item's gradients, rows in tile order
        const size_t head = (size_t)bh * N * kD;
        const int tok = tile_token(g, label, r);
        if (n > 0) {
            if (!warp_wait(smem_u32(&sm.bar_a), (P - 1) & 1, abortf, p.budget_ns)) return false;
            tc_fence_after();
            if (role == 1) {
                store_cols(tb + kColA0, p.dV + head, tok, col0, 1.0f);
                store_cols(tb + kColA1, p.dK + head, tok, col0, p.scale);
            } else {
                store_cols(tb + kColA0, p.dQ + head, tok, col0, p.scale);
            }
            tc_fence_before();  // the next item's first products overwrite the accumulators
        } else {
            float4* a = reinterpret_cast<float4*>((role == 1 ? p.dV : p.dQ) + head + (size_t)tok * kD + col0);
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (role == 1) {
                float4* b = reinterpret_cast<float4*>(p.dK + head + (size_t)tok * kD + col0);
#pragma unroll
                for (int i = 0; i < 4; ++i) b[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
}

__global__ void __launch_bounds__(kThreads, 2) ssba_bwd_ws_kernel(const __grid_constant__ WsMaps maps, const BwdParams p,
                                                               const int nk)
{
    WsSmem& sm = smem_layout();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        sm.abort_flag = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&sm.item_full[i]), 1);
            mbar_init(smem_u32(&sm.item_empty[i]), kCompute / 32 + kIssuers);
            mbar_init(smem_u32(&sm.ab_full[i]), 1);
            mbar_init(smem_u32(&sm.ab_empty[i]), kSdpIssuers);
        }
        for (int i = 0; i < kRing; ++i) {
            mbar_init(smem_u32(&sm.tile_full[i]), 1);
            mbar_init(smem_u32(&sm.tile_empty[i]), 1);
        }
        mbar_init(smem_u32(&sm.bar_s), kSdpIssuers);
        mbar_init(smem_u32(&sm.s_free), kCompute / 32);
        mbar_init(smem_u32(&sm.e_full), kCompute / 32);
        mbar_init(smem_u32(&sm.bar_a), 1);
        mbar_init(smem_u32(&sm.drain), kIssuers);
        fence_mbar_init();
    }
    for (int l = threadIdx.x; l < p.g.Tb(); l += kThreads) sm.win[l] = window_entry(p.g, l);
    if (warp == kProducer && lane < 16) {
        const CUtensorMap* m = lane < 4 ? &maps.q[lane] : lane < 8 ? &maps.k[lane - 4] : lane < 12 ? &maps.v[lane - 8]
                                                                                                  : &maps.o[lane - 12];
        tma_prefetch_desc(m);
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    bool ok = true;
    uint32_t P = 0;
    int kab = 0;
    if (p.withhold == 2 && threadIdx.x == kIssuer1 && blockIdx.x == 0) {
        // test hook: CTA 0's dP products start once another wait of the CTA has run out
        const uint64_t t0 = globaltimer_ns();
        while (!*static_cast<volatile int*>(&sm.abort_flag) && globaltimer_ns() - t0 < 4 * p.budget_ns) {
        }
    }
    if (warp < kCompute / 32)
        ok = compute(p, sm);
    else if (threadIdx.x == kIssuer0 || threadIdx.x == kIssuer1)
        ok = issue_sdp(p, sm, threadIdx.x == kIssuer1 ? 1 : 0);
    else if (threadIdx.x == kIssuer2)
        ok = issue_acc(p, sm);
    else if (warp == kProducer)
        ok = produce(maps, p, sm, nk, P, kab);
    // the flag as well as the verdicts: wait_phase returns none, and a phase that completes after its wait has
    // run out lets every later wait succeed. (Read behind the barrier: in front of it, the read makes the
    // whole kernel 7 to 10 % slower, 1024 px 132 -> 141 us.)
    const bool dead = __syncthreads_or(!ok) || *static_cast<volatile int*>(&sm.abort_flag);

    if (dead) {  // nothing more is issued: wait (bounded) for what is in flight, then report
        volatile int* abortf = &sm.abort_flag;
        *abortf = 1;
        if (warp == kProducer && lane == 0) {
            const uint64_t t0 = globaltimer_ns();
            auto settle = [&](uint32_t bar, uint32_t parity) {
                while (!mbar_try_wait(bar, parity) && globaltimer_ns() - t0 < p.budget_ns) {
                }
            };
            for (int i = 1; i <= 2 && i <= kab; ++i) settle(smem_u32(&sm.ab_full[(kab - i) & 1]), ((kab - i) >> 1) & 1);
            for (uint32_t i = 1; i <= (uint32_t)kRing && i <= P; ++i) {
                const uint32_t q = P - i;
                settle(smem_u32(&sm.tile_full[q % kRing]), (q / kRing) & 1);
            }
        }
        if (threadIdx.x == kIssuer0 || threadIdx.x == kIssuer1 || threadIdx.x == kIssuer2) {  // drain counts 3
            mma_commit(smem_u32(&sm.drain));
            const uint64_t t0 = globaltimer_ns();
            while (!mbar_try_wait(smem_u32(&sm.drain), 0) && globaltimer_ns() - t0 < p.budget_ns) {
            }
        }
        if (threadIdx.x == 0) atomicExch(p.status, SSBA_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(sm.tmem_base, kTmemCols);
}

}  // namespace

int launch_backward_ws(const ssba_desc& d, const Grid& g, int keep, float scale, const void* Q, const void* K,
                       const void* V, const void* O, const float* lse, const void* dO, const int32_t* idx,
                       const int32_t* cnt, float* dQ, float* dK, float* dV, void* workspace, cudaStream_t st,
                       uint64_t budget_ns, int withhold)
{
    if (d.head_dim != kD || g.blk != 8 || d.dtype != SSBA_BF16 || g.Tb() > 256 || (g.sr % 4) || (g.sc % 4))
        return SSBA_ERR_UNSUPPORTED;
    const int BH = d.B * d.heads;
    WsMaps maps;
    if (!encode_window_maps(maps.q, Q, BH, g.H, g.W) || !encode_window_maps(maps.k, K, BH, g.H, g.W) ||
        !encode_window_maps(maps.v, V, BH, g.H, g.W) || !encode_window_maps(maps.o, dO, BH, g.H, g.W))
        return SSBA_ERR_UNSUPPORTED;  // e.g. a base address the tensor maps cannot take
    const BwdLayout lay = bwd_layout(d, g, keep);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    BwdParams p;
    p.Q = static_cast<const __nv_bfloat16*>(Q);
    p.K = static_cast<const __nv_bfloat16*>(K);
    p.V = static_cast<const __nv_bfloat16*>(V);
    p.O = static_cast<const __nv_bfloat16*>(O);
    p.dO = static_cast<const __nv_bfloat16*>(dO);
    p.lse = lse;
    p.idx = idx;
    p.cnt = cnt;
    p.dQ = dQ;
    p.dK = dK;
    p.dV = dV;
    p.Dbuf = reinterpret_cast<float*>(ws);
    p.ctr = reinterpret_cast<int*>(ws + lay.ctr);
    p.toff = reinterpret_cast<int*>(ws + lay.toff);
    p.tcnt = reinterpret_cast<int*>(ws + lay.tcnt);
    p.tlist = reinterpret_cast<int*>(ws + lay.tlist);
    p.ld = reinterpret_cast<float4*>(ws + lay.ld);
    p.g = g;
    p.keep = keep;
    p.scale = scale;
    p.budget_ns = budget_ns;
    p.withhold = withhold;
    p.status = device_status_word();
    if (!p.status) {
        set_error("ssba_backward: could not resolve the device status word");
        return SSBA_ERR_CUDA;
    }
    static PerDeviceOnce attr;
    attr.run([] {
        cudaFuncSetAttribute(ssba_bwd_ws_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    });
    cudaError_t e = launch_bwd_rows(p, BH, st);
    if (e == cudaSuccess) {
        const int nk = BH * g.Tb();
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)std::min(2 * device_sm_count(), 2 * nk));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemBytes;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, ssba_bwd_ws_kernel, maps, p, nk);
    }
    if (e != cudaSuccess) {
        set_error("ssba_backward (persistent tensor-core kernel) launch: %s", cudaGetErrorString(e));
        return SSBA_ERR_CUDA;
    }
    return SSBA_OK;
}

}  // namespace ssba
