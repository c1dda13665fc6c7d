// select.cuh -- the Top-k gating of Sec. 2.2 / Algorithm 1 ("Top-k Smallest" dropped) on one
// row of affinities, shared by the mask kernels and the attention kernel's in-kernel
// selection, so that both keep bit-identical lists for the same scores.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ssba {
namespace sel {

// Order-preserving unsigned key of a float: larger key = larger value; -0.0 == +0.0.
__device__ __forceinline__ uint32_t order_key(float s)
{
    float f = s + 0.0f;  // -0.0 -> +0.0 so that equal values compare equal
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The float whose key is u.
__device__ __forceinline__ float key_value(uint32_t u)
{
    return __uint_as_float((u & 0x80000000u) ? (u ^ 0x80000000u) : ~u);
}

// Kept labels of one row, ascending, with the keys in registers (lane l holds the keys of labels
// l + 32 m, anything for labels >= Tb): the keep largest under the total order (S descending, label
// ascending), every path's rule, so the same scores give the same lists.
//   1. kPer of 8 and more (rows of more than 128 labels; where the keys pass through shared memory, more than
//      64): a threshold with exactly keep keys at or above it is looked for
//      between the row's smallest and largest value, each guess interpolated from the counts at the
//      two ends (and halfway where two guesses in a row moved the same end): about five counts for
//      random scores, a count being one ballot per 32 keys. Where there is one, the kept set is unique
//      and this is it.
//   2. Shorter rows, and otherwise (equal scores across the cut, infinities, NaN): an MSB-first radix
//      walk narrows the keys whose high bits equal a prefix to the group that holds the keep-th largest
//      key; keys above the group are kept, and within it the largest ones, the first equal ones in
//      label order. It stops once the group holds exactly the keys still to keep: about sixteen
//      counts, half of them over exponent bits that every score shares.
// Selection with the walk alone against both: 510 labels 83 -> 65 us, 256 labels 26 -> 24. With 64
// labels a count is two ballots and the code costs more than the counts: a 1024 px mask and forward 46.8
// us with the walk, 49.2 with both. (One key a lane: ballot_select<1> below.)
template <int kPer>
__device__ __forceinline__ void ballot_select(const uint32_t (&key)[kPer], int Tb, int keep, int lane, int32_t* dst)
{
    bool valid[kPer];
#pragma unroll
    for (int m = 0; m < kPer; ++m) valid[m] = lane + 32 * m < Tb;
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    if (kPer >= 8) {
#pragma unroll
        for (int m = 0; m < kPer; ++m)
            if (valid[m]) {
                kmin = min(kmin, key[m]);
                kmax = max(kmax, key[m]);
            }
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
    }
    uint32_t at = kmin;  // keys >= at are kept, if n == keep
    int n = Tb;
    const float inf = __uint_as_float(0x7f800000u);
    if (kPer >= 8 && n != keep && key_value(kmin) > -inf && key_value(kmax) < inf) {
        float lo = key_value(kmin), hi = key_value(kmax);  // n_lo >= keep keys at or above lo, n_hi < keep above hi
        int n_lo = Tb, n_hi = 0, moved = 0;
        for (int step = 0; step < 16; ++step) {
            const float f = (moved >= 2 || moved <= -2) ? 0.5f : __fdividef((float)(n_lo - keep) + 0.5f, (float)(n_lo - n_hi) + 1.f);
            const float mid = lo + (hi - lo) * f;
            at = order_key(mid);
            n = 0;
#pragma unroll
            for (int m = 0; m < kPer; ++m) n += __popc(__ballot_sync(0xffffffffu, valid[m] && key[m] >= at));
            if (n == keep) break;
            if (n > keep) {
                lo = mid;
                n_lo = n;
                moved = moved > 0 ? moved + 1 : 1;
            } else {
                hi = mid;
                n_hi = n;
                moved = moved < 0 ? moved - 1 : -1;
            }
        }
    }
    if (kPer >= 8 && n == keep) {
        int out = 0;
#pragma unroll
        for (int m = 0; m < kPer; ++m) {
            const bool kept = valid[m] && key[m] >= at;
            const uint32_t km = __ballot_sync(0xffffffffu, kept);
            if (kept) dst[out + __popc(km & ((1u << lane) - 1u))] = lane + 32 * m;
            out += __popc(km);
        }
        return;
    }
    uint32_t prefix = 0u, pmask = 0u;
    int remaining = keep, group = Tb;  // keys still to keep; keys whose bits under pmask equal prefix
    for (int bit = 31; bit >= 0 && group != remaining; --bit) {
        const uint32_t trial = prefix | (1u << bit), tmask = pmask | (1u << bit);
        int c = 0;
#pragma unroll
        for (int m = 0; m < kPer; ++m) c += __popc(__ballot_sync(0xffffffffu, valid[m] && (key[m] & tmask) == trial));
        if (c >= remaining) {
            prefix = trial;
            group = c;
        } else {
            remaining -= c;
            group -= c;
        }
        pmask = tmask;
    }
    int out = 0, eq_seen = 0;
#pragma unroll
    for (int m = 0; m < kPer; ++m) {
        const uint32_t hi = key[m] & pmask;
        const bool gt = valid[m] && hi > prefix, eq = valid[m] && hi == prefix;
        const uint32_t eqm = __ballot_sync(0xffffffffu, eq);
        const int eq_rank = eq_seen + __popc(eqm & ((1u << lane) - 1u));
        const bool kept = gt || (eq && eq_rank < remaining);
        const uint32_t km = __ballot_sync(0xffffffffu, kept);
        if (kept) dst[out + __popc(km & ((1u << lane) - 1u))] = lane + 32 * m;
        out += __popc(km);
        eq_seen += __popc(eqm);
    }
}

// Rows of up to 32 labels, one key a lane: its rank is counted over the others, read from their lanes. The
// reads do not wait for each other, where the counts of a walk do.
template <>
__device__ __forceinline__ void ballot_select<1>(const uint32_t (&key)[1], int Tb, int keep, int lane, int32_t* dst)
{
    int rank = 0;
#pragma unroll 8
    for (int k = 0; k < Tb; ++k) {
        const uint32_t other = __shfl_sync(0xffffffffu, key[0], k);
        rank += other > key[0] || (other == key[0] && k < lane);
    }
    const bool kept = lane < Tb && rank < keep;
    const uint32_t km = __ballot_sync(0xffffffffu, kept);
    if (kept) dst[__popc(km & ((1u << lane) - 1u))] = lane;
}

// Affinities S = q_b . k_b: four interleaved partial sums over d (components of 16-byte chunks, in
// chunk order), added as (a0 + a1) + (a2 + a3), for kRows rows of q and kKeys of k_b at once (each
// chunk is read once for all of them). q: row r at q + r * qld; chunk(k, c): key k's c-th chunk. Every
// path uses this order, so the same means give the same scores and lists. The pairs (a0, a1) and
// (a2, a3) go out as packed multiply-adds, with the roundings of single ones.
template <int kRows, int kKeys, class Chunk>
__device__ __forceinline__ void affinity_keys(float (&s)[kKeys][kRows], const float* q, int qld, Chunk chunk)
{
    float2 lo[kKeys][kRows], hi[kKeys][kRows];
#pragma unroll
    for (int k = 0; k < kKeys; ++k)
#pragma unroll
        for (int r = 0; r < kRows; ++r) lo[k][r] = hi[k][r] = make_float2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        float4 kv[kKeys];
#pragma unroll
        for (int k = 0; k < kKeys; ++k) kv[k] = chunk(k, c);
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const float4 v = *reinterpret_cast<const float4*>(q + r * qld + 4 * c);
#pragma unroll
            for (int k = 0; k < kKeys; ++k) {
                lo[k][r] = __ffma2_rn(make_float2(v.x, v.y), make_float2(kv[k].x, kv[k].y), lo[k][r]);
                hi[k][r] = __ffma2_rn(make_float2(v.z, v.w), make_float2(kv[k].z, kv[k].w), hi[k][r]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < kKeys; ++k)
#pragma unroll
        for (int r = 0; r < kRows; ++r) s[k][r] = (lo[k][r].x + lo[k][r].y) + (hi[k][r].x + hi[k][r].y);
}

template <int kRows, class Chunk>
__device__ __forceinline__ void affinity(float (&s)[kRows], const float* q, int qld, Chunk chunk)
{
    float t[1][kRows];
    affinity_keys<kRows, 1>(t, q, qld, [&](int, int c) { return chunk(c); });
#pragma unroll
    for (int r = 0; r < kRows; ++r) s[r] = t[0][r];
}

}  // namespace sel
}  // namespace ssba
