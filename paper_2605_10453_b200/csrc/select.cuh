// Selection of the k best (logit, id) pairs, shared by the streaming and the tensor-core path:
// warp-level bounds, ordering by counting, and the merge of split-V records.
// Records: 1 + k pairs of words per (row, slab): (maximum, sum of exp(logit - maximum)), then the slab's k
// (key, id) pairs in order.  Pair u of all P slabs of a row lie next to each other: the merge, whose lanes take
// a slab each, then reads whole lines.  (One record after the other it read a line per lane: eight rows took
// 2.2 us to load, 5120 lines through one SM's L1, against 1.3 us; records of 32-byte sectors 1.7 us.)
#pragma once
#include "ptx.cuh"
#include <float.h>

namespace slimspec {

static constexpr int kMaxK = 64;                      // largest k
static constexpr int kMergeCand = 192;                // candidates one row may park in the final merge
static constexpr int kMergeLists = 10;                // slab records a lane owns in the final merge
static constexpr int kMaxRecords = 32 * kMergeLists;  // records per row the merge can take
static constexpr int kNoId = 0x7fffffff;

// where pair u of slab s of a row lies
__host__ __device__ __forceinline__ size_t rec_row_pairs(int P, int k) { return (size_t)(1 + k) * P; }
__device__ __forceinline__ float2* rec_pair(float* part, int row, int P, int k, int s, int u)
{
    return reinterpret_cast<float2*>(part) + (size_t)row * rec_row_pairs(P, k) + (size_t)u * P + s;
}

// ------------------------------------------------------------------------------------------
// Selection.  Candidates are (key, id) with key = f2key(logit) and key 0 = none; the order is
// (key descending, id ascending).

// The k-th largest (k = 1..32) of the warp's 32 lane values, by counting: a lane's rank is the
// number of lanes ahead of it (larger key, or equal key and lower lane).
__device__ __forceinline__ uint32_t warp_kth_largest(uint32_t key, int k, int lane)
{
    int rank = 0;
#pragma unroll 4
    for (int s = 0; s < 32; ++s) {
        const uint32_t o = __shfl_sync(0xffffffffu, key, s);
        rank += (o > key || (o == key && s < lane)) ? 1 : 0;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, rank == k - 1);
    return __shfl_sync(0xffffffffu, key, __ffs(hit) - 1);
}

// A lower bound of the k-th largest of the warp's 32 lane values, by k rounds of "take the maximum out": exact unless
// values are equal (equal ones leave together, which only lowers the bound); 0 if there are fewer than k distinct ones.
// Cheaper than counting up to about a dozen.
__device__ __forceinline__ uint32_t warp_kth_rounds(uint32_t key, int k)
{
    uint32_t kth = 0u;
    for (int j = 0; j < k; ++j) {
        kth = warp_max_u32(key);
        key = key == kth ? 0u : key;
    }
    return kth;
}
__device__ __forceinline__ uint32_t warp_kth_largest_any(uint32_t key, int k, int lane)
{
    return k <= 12 ? warp_kth_rounds(key, k) : warp_kth_largest(key, k, lane);
}

// The same over 64 values, two per lane (value a has index lane, value b index lane + 32).
__device__ __forceinline__ uint32_t warp_kth_largest64(uint32_t a, uint32_t b, int k, int lane)
{
    int ra = 0, rb = 0;
#pragma unroll 4
    for (int s = 0; s < 32; ++s) {
        const uint32_t oa = __shfl_sync(0xffffffffu, a, s);
        const uint32_t ob = __shfl_sync(0xffffffffu, b, s);
        ra += (oa > a || (oa == a && s < lane)) ? 1 : 0;
        ra += (ob > a) ? 1 : 0;
        rb += (oa >= b) ? 1 : 0;
        rb += (ob > b || (ob == b && s < lane)) ? 1 : 0;
    }
    const unsigned hit_a = __ballot_sync(0xffffffffu, ra == k - 1);
    const unsigned hit_b = __ballot_sync(0xffffffffu, rb == k - 1);
    const uint32_t va = __shfl_sync(0xffffffffu, a, hit_a ? __ffs(hit_a) - 1 : 0);
    const uint32_t vb = __shfl_sync(0xffffffffu, b, hit_b ? __ffs(hit_b) - 1 : 0);
    return hit_a ? va : vb;
}

// A lower bound of the k-th largest (k <= 32 NV) of 32 NV keys, NV per lane, by bisection: at least k keys reach it, and
// no more where a value between the k-th and the next was met, as it nearly always is after eight or ten steps.
// (Ranks by counting every key against every other took 1000 to 1600 instructions for 128 and 160 keys.)
template <int NV>
__device__ __forceinline__ uint32_t warp_kth_bisect(const uint32_t (&key)[NV], int k)
{
    uint32_t mn = key[0], mx = key[0];
#pragma unroll
    for (int v = 1; v < NV; ++v) { mn = min(mn, key[v]); mx = max(mx, key[v]); }
    uint32_t lo = warp_min_u32(mn), hi = warp_max_u32(mx) + 1u;       // all keys reach lo, none hi
    while (hi - lo > 1u) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        int c = 0;
#pragma unroll
        for (int v = 0; v < NV; ++v) c += __popc(__ballot_sync(0xffffffffu, key[v] >= mid));
        if (c >= k) {
            lo = mid;
            if (c == k) break;
        } else {
            hi = mid;
        }
    }
    return lo;
}

// A candidate as one word: larger is better (key descending, id ascending).  0: none.
__device__ __forceinline__ unsigned long long cand_word(uint32_t key, int id)
{
    return ((unsigned long long)key << 32) | (uint32_t)~(uint32_t)id;
}
__device__ __forceinline__ uint32_t cand_key(unsigned long long c) { return (uint32_t)(c >> 32); }
__device__ __forceinline__ int cand_id(unsigned long long c) { return (int)~(uint32_t)c; }

// Sum of the values of the lanes before this one, and of all lanes.
__device__ __forceinline__ int warp_exclusive_sum(int v, int lane, int* total)
{
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, 31);
    return x - v;
}

// n distinct candidate words in shared memory (16-byte aligned, room for n + 3 words), in any order: the warp hands
// the min(n, k) best to put(rank, word), by counting: a candidate's rank is the number of better ones.
template <class Put>
__device__ __forceinline__ void warp_rank_words(unsigned long long* c, int n, int k, int lane, Put put)
{
    if (lane < 3) c[n + lane] = 0ull;          // the reads below go four at a time
    __syncwarp();
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        const unsigned long long mine = i < n ? c[i] : ~0ull;
        int rank = 0;
        for (int j = 0; j < n; j += 4) {
            const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(c + j);
            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(c + j + 2);
            rank += (a.x > mine) + (a.y > mine) + (b.x > mine) + (b.y > mine);
        }
        if (i < n && rank < k) put(rank, mine);
    }
    __syncwarp();
}

// is (ka, ia) strictly after (kb, ib) in the order, i.e. a worse candidate?
__device__ __forceinline__ bool after(uint32_t ka, int ia, uint32_t kb, int ib)
{
    return ka < kb || (ka == kb && ia > ib);
}
// is (ka, ia) a better candidate than (kb, ib)?
__device__ __forceinline__ bool better(uint32_t ka, int ia, uint32_t kb, int ib)
{
    return ka > kb || (ka == kb && ia < ib);
}

// ------------------------------------------------------------------------------------------
// One task of the merge, run by one warp: kind 0 = the row's log-sum-exp from the records'
// (maximum, sum-exp) pairs, written to *lse_out; kind 1 = its k best entries, in order, to out, padded
// with empty ones (key 0).  A lane owns the records lane, lane + 32, ... (NL of them at most) and keeps what it loads
// in registers: one round trip to the L2.  area: kMergeWarpBytes of shared memory of this warp, 16-byte aligned.
static constexpr int kMergeWarpBytes = (kMergeCand + 4) * 8 + 16;
template <int NL>
__device__ __forceinline__ void merge_task(const float* part, int P, int k, int row, int kind, int lane, float* lse_out,
                                           unsigned long long* out, unsigned char* area)
{
    const float2* rows = reinterpret_cast<const float2*>(part) + (size_t)row * rec_row_pairs(P, k);
    if (kind == 0) {
        float2 ms[NL];
#pragma unroll
        for (int q = 0; q < NL; ++q) {
            const int s = lane + 32 * q;
            ms[q] = s < P ? __ldcg(rows + s) : make_float2(-FLT_MAX, 0.f);
        }
        float gm = -FLT_MAX;
#pragma unroll
        for (int q = 0; q < NL; ++q) gm = fmaxf(gm, ms[q].x);
        gm = warp_max(gm);
        float gs = 0.f;
#pragma unroll
        for (int q = 0; q < NL; ++q) gs += ms[q].y * __expf(ms[q].x - gm);
        gs = warp_sum(gs);
        if (lane == 0) *lse_out = gm + __logf(gs);
        return;
    }
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(area);
    int* cnt = reinterpret_cast<int*>(cand + kMergeCand + 4);
    // the first three entries of every record, then the bound
    const float2 none = make_float2(0.f, __int_as_float(kNoId));
    float2 e0[NL], e1[NL], e2[NL];
#pragma unroll
    for (int q = 0; q < NL; ++q) {
        const int s = lane + 32 * q;
        e0[q] = s < P ? __ldcg(rows + P + s) : none;
        e1[q] = s < P && k >= 2 ? __ldcg(rows + 2 * P + s) : none;
        e2[q] = s < P && k >= 3 ? __ldcg(rows + 3 * P + s) : none;
    }
    // Up to k = 24 the k-th largest of the lanes' best entries: with 24 of 32 lanes about 44 entries reach it.
    // Beyond, every record's best entry counts by itself (k = 64 of 148 records: about 84 entries).
    uint32_t kth;
    if (k <= 24) {
        uint32_t hk[1] = {0u};
#pragma unroll
        for (int q = 0; q < NL; ++q) hk[0] = max(hk[0], __float_as_uint(e0[q].x));
        kth = k <= 12 ? warp_kth_rounds(hk[0], k) : warp_kth_bisect<1>(hk, k);
    } else {
        uint32_t hk[NL];
#pragma unroll
        for (int q = 0; q < NL; ++q) hk[q] = __float_as_uint(e0[q].x);
        kth = warp_kth_bisect<NL>(hk, k);
    }
    kth = max(kth, 1u);                      // empty entries (key 0) never count
    // the entries that reach the bound, by ballot: the first ones, then, where any do, the second and third ones (a record's
    // list is in order, so its later entries matter only where the earlier ones reach the bound)
    const unsigned below = (1u << lane) - 1u;
    int n = 0;
    bool second = false, third = false;
    auto park = [&](float2 e) {
        const bool in = __float_as_uint(e.x) >= kth;
        const unsigned b = __ballot_sync(0xffffffffu, in);
        const int pos = n + __popc(b & below);
        if (in && pos < kMergeCand) cand[pos] = cand_word(__float_as_uint(e.x), __float_as_int(e.y));
        n += __popc(b);
    };
#pragma unroll
    for (int q = 0; q < NL; ++q) { park(e0[q]); second = second || __float_as_uint(e1[q].x) >= kth; }
    if (__any_sync(0xffffffffu, second)) {
#pragma unroll
        for (int q = 0; q < NL; ++q) { park(e1[q]); third = third || __float_as_uint(e2[q].x) >= kth; }
        if (__any_sync(0xffffffffu, third)) {
            if (lane == 0) *cnt = n;
            __syncwarp();
#pragma unroll 1
            for (int s = lane; s < P; s += 32) {
                for (int j = 2; j < k; ++j) {
                    const float2 en = __ldcg(rows + (size_t)(1 + j) * P + s);
                    const uint32_t kj = __float_as_uint(en.x);
                    if (kj < kth) break;
                    const int at = atomicAdd(cnt, 1);
                    if (at < kMergeCand) cand[at] = cand_word(kj, __float_as_int(en.y));
                }
            }
            __syncwarp();
            n = *cnt;
        }
    }
    __syncwarp();
    if (n <= kMergeCand) {
        warp_rank_words(cand, n, k, lane, [&](int rank, unsigned long long c) { out[rank] = c; });
        for (int j = n + lane; j < k; j += 32) out[j] = cand_word(0u, kNoId);
    } else {
        // slow path: k rounds over every entry of the row's records, each round taking the best
        // entry after the previous winner
        uint32_t lk = 0xffffffffu;
        int li = -1;
        for (int j = 0; j < k; ++j) {
            uint32_t bk = 0u;
            int bi = kNoId;
            for (int s = lane; s < P; s += 32) {
                for (int e = 0; e < k; ++e) {
                    const float2 en = __ldcg(rows + (size_t)(1 + e) * P + s);
                    const uint32_t ke = __float_as_uint(en.x);
                    const int ie = __float_as_int(en.y);
                    if (ke == 0u || !better(ke, ie, bk, bi)) break;        // the list is in order: nothing better follows ...
                    if (after(ke, ie, lk, li)) { bk = ke; bi = ie; break; }  // ... and the first one after the winner is its best
                }
            }
            const uint32_t wk = warp_max_u32(bk);
            const uint32_t wi = warp_min_u32(bk == wk ? (uint32_t)bi : 0xffffffffu);
            lk = wk;
            li = (int)wi;
            if (lane == 0) out[j] = cand_word(wk, wk != 0u ? (int)wi : kNoId);
            if (wk == 0u) { lk = 0u; li = kNoId; }
        }
    }
}

}  // namespace slimspec
