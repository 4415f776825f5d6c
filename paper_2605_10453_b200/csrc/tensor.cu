// Tensor-core path for larger M: out = X W with X[M][K] (rows on the MMA's M side, K-major) and
// W[K][N] (N-major), bf16 inputs, fp32 accumulation in tensor memory (tcgen05).
//   down-projection  z = h A      X = h, W = A, K split over the CTAs of a cluster, which add their tiles up
//   up-projection    logits = z B X = z (bf16), W = B, fused online log-softmax / top-k epilogue
//   full-rank head   logits = h W X = h, W = W, same epilogue
// (Section 4.1; the softmax of Section 3.2 and the candidate selection.)
//
// One CTA per SM: one warp feeds a ring of shared-memory stages by TMA, one thread of another
// warp issues the MMAs into one of two accumulator buffers in tensor memory, eight epilogue warps read the
// finished buffer (a thread per row and column half) and keep that row's running max / sum-exp / top-k while
// the next tile's MMAs run.
#include "kernels.h"
#include "ptx.cuh"
#include "select.cuh"
#include "tmap.h"
#include <float.h>
#include <string.h>

namespace slimspec {

static constexpr int kTcRows = 128;          // rows of a tile that one CTA has
static constexpr int kTcKChunk = 64;         // K per stage: 64 bf16 = one 128-byte swizzle row
// Twelve warps.  A warp reads only the lane quarter (warp id mod 4) of tensor memory and warps are
// dealt to the SM's four schedulers by the same rule, so the rows of quarter q are worked on by the
// scheduler q.  Epilogue warps 0..7 (two a quarter, half of the columns each); the loading and the issuing warp sit with the
// quarters that fill last.
static constexpr int kTcThreads = 384;
static constexpr int kTcEpiWarps = 8, kTcLoadWarp = 10, kTcMmaWarp = 11;
static constexpr int kTcMaxK = 32;           // largest k
static constexpr int kTcList = 48;           // candidates a row parks before the list is compacted
static constexpr int kTcListPitch = 49;      // entries between two rows' lists in shared memory: odd, so lanes hit distinct banks
static constexpr int kTcEpiThreads = kTcEpiWarps * 32;
// shared memory the final sort of the lists needs (values and ids of every epilogue thread)
static constexpr size_t kTcSortBytes = (size_t)kTcEpiThreads * kTcListPitch * 8;
static constexpr int kTcMaxStages = 8;
static constexpr int kTcMaxResident = 16;    // most K chunks of a resident X
static constexpr int kTcPartPitch = 132;     // floats between two rows of a partial tile in shared memory: 33 16-byte units, odd
static constexpr int kTcBoundPolls = 32;     // looks at the other CTAs' maxima after the first tile
static constexpr float kLog2e = 1.4426950408889634f;

struct alignas(64) TcParams {
    CUtensorMap mapX;       // X[M][K]: box 64 (K) x rows, 128-byte swizzle
    CUtensorMap mapW;       // W[K][N]: box 64 (N) x 64 (K), 128-byte swizzle
    CUtensorMap mapX2;      // split mode: the low part of X, same shape and box as mapX
    int M, N;
    int nrb, nct;           // row blocks (128 rows a CTA), column tiles
    int nks;                // mode 2: K splits = CTAs of a cluster
    int chunks;             // K chunks of 64 (the last one may run past K: zeros)
    int gct;                // CTAs (pairs) that share a row block; column tiles go round-robin
    int mode;               // 0: top-k records, 1: fp32 out[M][N], 2: bf16 code
    int k;
    int ns;                 // stages of the ring
    int xbox_bytes;         // bytes of one X box: (rows of the box, 8..128) x 128; rows past the box are garbage in,
                            // garbage out, and belong to no live row
    int split;              // 1: X = X_hi + X_lo (two bf16 matrices): two MMAs per step into one accumulator
    int xres;               // 1: the row block's whole X is loaded once and stays in shared memory; else it travels with the stages
    float* out;             // mode 1
    float* part;            // records of 2 gct slabs a row (see select.cuh): two column halves per CTA
    unsigned long long* bound;   // mode 0: [k][bound_pitch] words (call number, key), see bound_publish
    int bound_pitch;
    unsigned int epoch;     // number of the call: larger than every earlier one's, never 0
    bf16* z[3];             // mode 2: the code [M][z_pitch] and, if not null, its rounding remainder and what the two leave
    int z_pitch;
    int* err;
};

// A row's candidate list: up to kTcList (value, id) pairs above the row's threshold, appended in
// the order the columns arrive (ascending id).  topk_compact sorts the list (values descending,
// equal values keep their order, i.e. lower id first), cuts it to the k best and returns the
// new threshold: the k-th value if the list holds k entries, else the old bound.
__device__ __noinline__ float topk_compact(uint2* list, int& cnt, int k, float thr0)
{
    for (int i = 1; i < cnt; ++i) {
        const uint2 v = list[i];
        int pos = i;
        while (pos > 0 && __uint_as_float(list[pos - 1].x) < __uint_as_float(v.x)) {
            list[pos] = list[pos - 1];
            --pos;
        }
        list[pos] = v;
    }
    if (cnt > k) cnt = k;
    return cnt == k ? __uint_as_float(list[k - 1].x) : thr0;
}

__device__ __forceinline__ float ex2_fast(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The bound below a row's k-th largest logit that keeps the candidate lists short.  The (CTA, column half) pairs that
// work on a row are dealt to k groups; each adds the maximum of the columns it has seen so far to its group's word.  The
// groups' columns are disjoint, so the smallest of the k words is reached by k logits of the row.  A word is (call
// number, key) and is only ever raised: what earlier calls left is overruled by the number, nothing is cleared and
// nobody waits for anybody; a word without this call's number only means that there is no bound yet.
__device__ __forceinline__ void bound_publish(const TcParams& p, int group, int m, float mx)
{
    const unsigned long long w = ((unsigned long long)p.epoch << 32) | f2key(mx);
    asm volatile("red.relaxed.gpu.global.max.u64 [%0], %1;" ::"l"(p.bound + (size_t)group * p.bound_pitch + m), "l"(w) : "memory");
}
// Largest float that is certainly below the k-th largest logit, or -FLT_MAX.
__device__ __noinline__ float bound_read(const unsigned long long* bound, int pitch, unsigned int epoch, int k, int m)
{
    uint32_t lo = 0xffffffffu;
#pragma unroll 8
    for (int g = 0; g < k; ++g) {
        unsigned long long w;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(bound + (size_t)g * pitch + m) : "memory");
        lo = min(lo, (uint32_t)(w >> 32) == epoch ? (uint32_t)w : 0u);
    }
    const float v = key2f(lo);
    if (lo <= f2key(-FLT_MAX)) return -FLT_MAX;
    return v == 0.f ? -__uint_as_float(1u) : key2f(lo - 1u);       // -0 and +0 compare equal: the next value below both
}

// What one epilogue thread carries for its row across the tiles of its CTA.
struct EpiRow {
    float run_max, run_sum;     // online softmax: maximum so far, sum of exp(logit - maximum)
    float thr;                  // candidates must beat this
    int cnt;                    // candidates parked in the list
};

// Eight columns of one row: those above the threshold are parked.  (No branch but for a list that may not take eight more.)
__device__ __forceinline__ void epi_park(const float* x, int col, int k, EpiRow& st, uint2* list)
{
    if (st.cnt > kTcList - 8) {
        int c = st.cnt;      // a copy: the state stays in registers
        st.thr = fmaxf(st.thr, topk_compact(list, c, k, st.thr));
        st.cnt = c;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (x[e] > st.thr) list[st.cnt++] = make_uint2(__float_as_uint(x[e]), (uint32_t)(col + e));
    }
}

// 32 consecutive columns of one row: maximum and sum of exp and, with PARK, the candidates.  Columns from nvalid on (last
// tile only) count as -FLT_MAX.
__device__ __forceinline__ void epi_chunk(const uint32_t (&v)[32], int nvalid, int col, int k, bool park, EpiRow& st, uint2* list)
{
    float x[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) x[e] = __uint_as_float(v[e]);
    if (nvalid < 32) {
#pragma unroll
        for (int e = 0; e < 32; ++e) x[e] = e < nvalid ? x[e] : -FLT_MAX;
    }
    float m8[4];       // maxima of the four groups of eight columns (three-input max: four steps a group)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float g = max3(x[q * 8], x[q * 8 + 1], x[q * 8 + 2]);
        g = max3(g, x[q * 8 + 3], x[q * 8 + 4]);
        g = max3(g, x[q * 8 + 5], x[q * 8 + 6]);
        m8[q] = fmaxf(g, x[q * 8 + 7]);
    }
    const float cmax = fmaxf(max3(m8[0], m8[1], m8[2]), m8[3]);
    if (cmax > st.run_max) {
        st.run_sum *= ex2_fast((st.run_max - cmax) * kLog2e);
        st.run_max = cmax;
    }
    // sum of 2^(x log2(e) - max log2(e)): the scaling and the adds go two columns an instruction
    const float nmb = -st.run_max * kLog2e;
    const float2 sc = make_float2(kLog2e, kLog2e), of = make_float2(nmb, nmb);
    float2 sacc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        const float2 t = __ffma2_rn(make_float2(x[e], x[e + 1]), sc, of);
        sacc[(e >> 1) & 1] = __fadd2_rn(sacc[(e >> 1) & 1], make_float2(ex2_fast(t.x), ex2_fast(t.y)));
    }
    st.run_sum += (sacc[0].x + sacc[0].y) + (sacc[1].x + sacc[1].y);
    // Some row of the warp has a candidate in most chunks, but a given group of eight rarely has one of any row.
    if (park && __any_sync(0xffffffffu, cmax > st.thr)) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (__any_sync(0xffffffffu, m8[q] > st.thr)) epi_park(x + q * 8, col + q * 8, k, st, list);
    }
}

// ------------------------------------------------------------------------------------------
// CG: CTAs that work on one tile (1: 128 rows x NV columns; 2: a pair of CTAs, 256 rows x NV columns, 128 rows in each
// CTA's tensor memory; each loads its rows of X and half of the columns of W).
template <int CG, int NV>
__global__ void __launch_bounds__(kTcThreads, 1) k_tc_gemm(const __grid_constant__ TcParams p)
{
    constexpr int WBOX_BYTES = kTcKChunk * 64 * 2;          // 8 KB: 64 k x 64 columns
    constexpr int WCOLS = NV / CG;                          // columns of W that this CTA loads
    constexpr int W_BYTES = WBOX_BYTES * (WCOLS / 64);
    const int NS = p.ns;
    const bool xres = p.xres != 0, split = p.split != 0;
    const int XH = p.xbox_bytes;                            // one X box (high or low part) of a K chunk
    const int XB = split ? 2 * XH : XH;                     // X bytes per K chunk: high part, then low part
    const int SB = xres ? W_BYTES : XB + W_BYTES;           // a stage: X (unless it is resident), then W
    // instruction descriptor: D fp32, A and B bf16, A K-major, B MN-major, N = NV, M = 128 CG
    constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (0u << 15) | (1u << 16) |
                               ((uint32_t)(NV >> 3) << 17) | ((uint32_t)((CG * kTcRows) >> 4) << 24);

    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t full[kTcMaxStages], empty[kTcMaxStages], acc_full[2], acc_empty[2], x_full[kTcMaxResident];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    unsigned char* xarea = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    volatile int* abort_flag = &abort_s;

    // The warp's number and the base in tensor memory come from lane 0: the compiler then knows them to be the same in all lanes
    // and keeps the operands of tensor-core and TMA instructions in uniform registers.
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    // which tile: the CTAs of a pair (mode 2: of a K split) are neighbours
    const int per = CG == 2 ? 2 : p.nks;
    const int rank = (int)blockIdx.x % per, rest = (int)blockIdx.x / per;
    const int ks = CG == 2 ? 0 : rank;
    const int rb = CG == 2 ? (rest % p.nrb) * 2 + rank : rest % p.nrb;      // row block of 128 rows
    const int cg = rest / p.nrb;                            // position among the CTAs (pairs) of this row block
    const int ntiles = cg < p.nct ? (p.nct - cg + p.gct - 1) / p.gct : 0;
    const int c0 = ks * p.chunks / p.nks, cps = (ks + 1) * p.chunks / p.nks - c0;
    unsigned char* stages = xarea + (xres ? (size_t)cps * XB : 0);

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], CG * kTcEpiWarps); }
        for (int c = 0; c < kTcMaxResident; ++c) mbar_init(&x_full[c], 1);
        abort_s = 0;
        mbar_fence_init();
        prefetch_tensor_map(&p.mapX);
        prefetch_tensor_map(&p.mapW);
        if (p.split) prefetch_tensor_map(&p.mapX2);
    }
    if (warp == kTcMmaWarp) {
        if (CG == 2) tmem_alloc_pair(&tmem_base_s, 2 * NV);
        else tmem_alloc(&tmem_base_s, 2 * NV);
    }
    tc_fence_before_sync();
    if (CG == 2) cluster_sync();
    else __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    // Everything above touched no global data: under programmatic dependent launch it overlaps the kernel before.  That
    // kernel's results are needed for X, and what the epilogue writes belongs to it until it has finished; the
    // weights are final before the call is made, so the first stages' are sent for at once.
    pdl_launch_dependents();

    if (warp == kTcLoadWarp) {
        // ================= producer =================
        // Barriers of a pair are the first CTA's: it expects the bytes of both.
        const uint32_t full0 = CG == 2 ? cluster_map(smem_u32(&full[0]), 0) : smem_u32(&full[0]);
        const uint32_t xfull0 = CG == 2 ? cluster_map(smem_u32(&x_full[0]), 0) : smem_u32(&x_full[0]);
        const bool first_cta = CG == 1 || rank == 0;
        auto load = [&](unsigned char* dst, const CUtensorMap* map, int x, int y, uint32_t bar0, uint64_t* bar_here) {
            if (CG == 2) tma_load_2d_pair(dst, map, x, y, bar0);
            else tma_load_2d(dst, map, x, y, bar_here);
        };
        auto send_x = [&](unsigned char* dst, int c, uint32_t bar0, uint64_t* bar_here) {
            load(dst, &p.mapX, (c0 + c) * kTcKChunk, rb * kTcRows, bar0, bar_here);
            if (split) load(dst + XH, &p.mapX2, (c0 + c) * kTcKChunk, rb * kTcRows, bar0, bar_here);
        };
        auto send_w = [&](int s, int ct, int c) {
            if (first_cta) mbar_arrive_expect_tx(&full[s], (uint32_t)(CG * SB));
            unsigned char* st = stages + (size_t)s * SB + (xres ? 0 : XB);
#pragma unroll
            for (int i = 0; i < WCOLS / 64; ++i)
                load(st + i * WBOX_BYTES, &p.mapW, ct * NV + (CG == 2 ? rank * WCOLS : 0) + i * 64, (c0 + c) * kTcKChunk, full0 + (uint32_t)(s * 8), &full[s]);
        };
        const int total = ntiles * cps, npre = total < NS ? total : NS;
        if (elect_one()) {
            for (int i = 0; i < npre; ++i) send_w(i, cg + (i / cps) * p.gct, i % cps);
        }
        __syncwarp();
        pdl_wait();
        if (xres && ntiles > 0 && elect_one()) {
            for (int c = 0; c < cps; ++c) {
                if (first_cta) mbar_arrive_expect_tx(&x_full[c], (uint32_t)(CG * XB));
                send_x(xarea + (size_t)c * XB, c, xfull0 + (uint32_t)(c * 8), &x_full[c]);
            }
        }
        __syncwarp();
        // ring positions are kept as (slot, phase) pairs: no division on this path
        int s = 0, ph = 0, i = 0;
        bool alive = true;
        for (int t = 0; t < ntiles; ++t) {
            for (int c = 0; c < cps; ++c, ++i) {
                if (i >= npre && alive) alive = mbar_wait_uniform(&empty[s], ph ^ 1);
                if (alive) {
                    if (elect_one()) {
                        if (i >= npre) send_w(s, cg + t * p.gct, c);
                        if (!xres) send_x(stages + (size_t)s * SB, c, full0 + (uint32_t)(s * 8), &full[s]);
                    }
                    __syncwarp();
                }
                if (++s == NS) { s = 0; ph ^= 1; }
            }
        }
        // the last lap's stages come free before this CTA's shared memory goes
        for (int u = total - npre; u < total && alive; ++u) alive = mbar_wait_uniform(&empty[u % NS], (u / NS) & 1);
        if (!alive) mbar_gave_up(abort_flag, p.err, ERR_WAIT_EMPTY);
    } else if (warp == kTcMmaWarp) {
        // ================= MMA issuer =================
        // What counts here is the time an instruction takes to issue: in a loop of one lane, or one whose end the compiler cannot
        // tell to be the same in all lanes, every operand goes through a move to a uniform register, and an MMA took
        // 90 to 120 cycles (of the 64 to 128 its arithmetic takes), a chunk 600 to 800.  So the warp runs the loop
        // together, no exit depends on a lane, and one lane is elected at each issue.  Descriptors are running low words
        // (start address and leading offset; the high word is the same for every operand).
        if (CG == 1 || rank == 0) {
            constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);     // SBO 1024, version 1, 128-byte swizzle
            const uint32_t ring_w = (smem_u32(stages) >> 4) & 0x3fffu, SBW = (uint32_t)SB >> 4;
            const uint32_t xres_w = ((smem_u32(xarea) >> 4) & 0x3fffu) | (1u << 16);                       // LBO 16
            const uint32_t a_step = (uint32_t)XB >> 4, a_lowpart = (uint32_t)XH >> 4;
            int s = 0, ph = 0;
            uint32_t st = ring_w;
            bool alive = true;
            pdl_wait();          // nothing to do before X is there, and the waits below are bounded
            for (int t = 0; t < ntiles; ++t) {
                const int buf = t & 1;
                if (t >= 2 && alive) alive = mbar_wait_uniform(&acc_empty[buf], ((t >> 1) - 1) & 1);
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * NV);
                uint32_t xr = xres_w;
                for (int c = 0; c < cps; ++c) {
                    if (t == 0 && xres && alive) alive = mbar_wait_uniform(&x_full[c], 0);
                    if (alive) alive = mbar_wait_uniform(&full[s], ph);
                    const uint32_t a_lo = xres ? xr : st | (1u << 16);
                    const uint32_t b_lo = (st + (xres ? 0u : a_step)) | ((uint32_t)(WBOX_BYTES >> 4) << 16);
                    if (alive) {
                        if (elect_one()) {
                            // 16 of K per instruction: 32 bytes along a K-major row of X, two 8-row groups of the N-major W tile
                            auto mma = [&](uint32_t a, uint32_t b, uint32_t acc) {
                                if (CG == 2) tc_mma_bf16_words_pair(d_tmem, a, b, DESC_HI, IDESC, acc);
                                else tc_mma_bf16_words(d_tmem, a, b, DESC_HI, IDESC, acc);
                            };
#pragma unroll
                            for (int j = 0; j < kTcKChunk / 16; ++j) mma(a_lo + (uint32_t)(j * 2), b_lo + (uint32_t)(j * 128), j > 0 || c > 0 ? 1u : 0u);
                            if (split) {
#pragma unroll
                                for (int j = 0; j < kTcKChunk / 16; ++j) mma(a_lo + a_lowpart + (uint32_t)(j * 2), b_lo + (uint32_t)(j * 128), 1u);
                            }
                            if (CG == 2) tc_commit_pair(&empty[s]);
                            else tc_commit(&empty[s]);
                            if (c == cps - 1) {
                                if (CG == 2) tc_commit_pair(&acc_full[buf]);
                                else tc_commit(&acc_full[buf]);
                            }
                        }
                        __syncwarp();
                    }
                    xr += a_step;
                    st += SBW;
                    if (++s == NS) { s = 0; ph ^= 1; st = ring_w; }
                }
            }
            if (!alive) mbar_gave_up(abort_flag, p.err, ERR_WAIT_FULL);
        }
    } else if (warp < kTcEpiWarps) {
        // ================= epilogue: thread = row =================
        pdl_wait();
        const int quarter = warp & 3;                        // the lane quarter this warp may read
        const int half = warp >> 2;                          // two warps share a quarter: each takes half the columns
        const int row = quarter * 32 + lane;
        const int m = rb * kTcRows + row;
        const bool live = m < p.M, warp_live = rb * kTcRows + quarter * 32 < p.M;
        const int k = p.k;
        const uint32_t acc_empty0 = CG == 2 ? cluster_map(smem_u32(&acc_empty[0]), 0) : smem_u32(&acc_empty[0]);
        EpiRow st;
        st.run_max = -FLT_MAX;
        st.run_sum = 0.f;
        st.cnt = 0;
        st.thr = live ? -FLT_MAX : __int_as_float(0x7f800000);       // rows past M have no candidates
        uint2 list[kTcList];
        const int group = (2 * cg + half) % k;
        bool alive = true;
        for (int t = 0; t < ntiles && alive; ++t) {
            const int buf = t & 1;
            const int colbase = (cg + t * p.gct) * NV + half * (NV / 2);
            if (p.mode == 0 && live && t >= 1 && (t & (t - 1)) == 0) st.thr = fmaxf(st.thr, bound_read(p.bound, p.bound_pitch, p.epoch, k, m));
            if (!mbar_wait_warp(&acc_full[buf], (t >> 1) & 1, abort_flag, p.err, ERR_WAIT_ACC)) { alive = false; break; }
            tc_fence_after_sync();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * NV + half * (NV / 2));
            // The warp has read what it needs of the buffer.
            auto hand_back = [&] {
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    if (CG == 2) mbar_arrive_cluster(acc_empty0 + (uint32_t)(buf * 8));
                    else mbar_arrive(&acc_empty[buf]);
                }
            };
            const int ncol = warp_live ? min(NV / 2, p.N - colbase) : 0;      // the warp's columns of this tile; may be negative
            if (NV >= 128 && p.mode == 0 && ncol > 0) {
#pragma unroll 1
                for (int i = 0; i < ncol; i += 64) {
                    uint32_t v[32], w[32];
                    tmem_ld_32x32(taddr + (uint32_t)i, v);
                    tmem_ld_32x32(taddr + (uint32_t)i + 32, w);
                    tmem_ld_wait();
                    // The next MMAs into this buffer start while the last columns are worked on (handed back before the last 64
                    // of them rather than 32: 512 rows 86.3 -> 83.2 us, 128 rows 54.8 -> 51.4).
                    if (i + 64 >= ncol && t > 0) hand_back();
                    epi_chunk(v, ncol - i, colbase + i, k, t > 0, st, list);
                    if (i + 32 < ncol) epi_chunk(w, ncol - i - 32, colbase + i + 32, k, t > 0, st, list);
                }
                if (((t + 1) & t) == 0 && live) bound_publish(p, group, m, st.run_max);
                if (t == 0) {
                    // The other CTAs' first maxima are out at about the same time; the next tile's MMAs run meanwhile.
                    int polls = 0;
                    float b = -FLT_MAX;
                    do {
                        if (live) b = bound_read(p.bound, p.bound_pitch, p.epoch, k, m);
                    } while (++polls < kTcBoundPolls && 2 * p.gct >= k && __any_sync(0xffffffffu, live && b == -FLT_MAX));
                    st.thr = fmaxf(st.thr, b);
                    // with the bound, the first tile once more, for its candidates
#pragma unroll 1
                    for (int g = 0; g < ncol / 8; ++g) {
                        uint32_t w[8];
                        tmem_ld(taddr + (uint32_t)(g * 8), w);
                        tmem_ld_wait();
                        float x[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(w[e]);
                        epi_park(x, colbase + g * 8, k, st, list);
                        __syncwarp();
                    }
                    hand_back();
                }
                continue;
            }
            if (p.mode == 1) {
                float* dst = p.out + (size_t)m * p.N + colbase;
#pragma unroll 1
                for (int i = 0; i < ncol; i += 32) {
                    uint32_t v[32];
                    tmem_ld_32x32(taddr + (uint32_t)i, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; e += 8) {
                        if (live && i + e < ncol) st_global_v8(dst + i + e, v + e);      // N is a multiple of 8, so a group of eight is all in or all out
                    }
                }
            } else if (p.mode == 2) {
                // the partial tile, to shared memory: every MMA has completed, the ring is idle
                float* dst = reinterpret_cast<float*>(xarea) + (size_t)row * kTcPartPitch + half * (NV / 2);
#pragma unroll 1
                for (int i = 0; i < ncol; i += 32) {
                    uint32_t v[32];
                    tmem_ld_32x32(taddr + (uint32_t)i, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<float4*>(dst + i + e) = make_float4(__uint_as_float(v[e]), __uint_as_float(v[e + 1]), __uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
                }
            }
            hand_back();
        }
        if (alive && live && p.mode == 0 && ntiles > 0) {
            // The lists live in local memory, which this kernel's small L1 hardly caches.  Every MMA has completed by
            // now (the last accumulator was handed over), so the operand rings are dead: the list is put in order there, an
            // entry's place being the number of better ones (of equal values the earlier has the lower id).
            uint2* sl = reinterpret_cast<uint2*>(xarea) + (size_t)(warp * 32 + lane) * kTcListPitch;
            const int cnt = st.cnt;
            for (int j = 0; j < cnt; ++j) sl[j] = list[j];
            const int P = 2 * p.gct, slab = 2 * cg + half;
            *rec_pair(p.part, m, P, k, slab, 0) = make_float2(st.run_max, st.run_sum);
            for (int j = 0; j < cnt; ++j) {
                const uint2 mine = sl[j];
                int rank = 0;
#pragma unroll 4
                for (int i = 0; i < cnt; ++i) {
                    const float o = __uint_as_float(sl[i].x);
                    rank += o > __uint_as_float(mine.x) || (o == __uint_as_float(mine.x) && i < j) ? 1 : 0;
                }
                // (key, id) pairs; -0 and +0 rank alike
                if (rank < k) *rec_pair(p.part, m, P, k, slab, 1 + rank) = make_float2(__uint_as_float(f2key(__uint_as_float(mine.x) + 0.f)), __int_as_float((int)mine.y));
            }
            // the merge looks at the first three and then on to the first empty one
            const int nw = min(k, max(cnt + 1, 3));
            for (int j = cnt; j < nw; ++j) *rec_pair(p.part, m, P, k, slab, 1 + j) = make_float2(__uint_as_float(0u), __int_as_float(kNoId));
        }
    }
    // ---- teardown: every role is past its last use of tensor memory
    tc_fence_before_sync();
    __syncwarp();
    if (CG == 2) cluster_sync_exec();       // nothing in shared memory is handed over, and the release takes a microsecond
    else if (p.nks > 1) cluster_sync();
    else __syncthreads();
    tc_fence_after_sync();
    if (warp == kTcMmaWarp) {
        if (CG == 2) tmem_dealloc_pair(tmem_base, 2 * NV);
        else tmem_dealloc(tmem_base, 2 * NV);
    }
    if (CG == 1 && NV <= 128 && p.mode == 2) {
        // The code: CTA ks of the cluster adds the partial tiles of its share of the rows, in the order of K, rounds the
        // sum to bf16 and keeps the rounding remainder as a second matrix where the caller wants it.
        const int r0 = ks * kTcRows / p.nks, nr = (ks + 1) * kTcRows / p.nks - r0;
        const int col0 = cg * NV;
        const uint32_t area = smem_u32(xarea);
        for (int e = tid; e < nr * (NV / 4); e += kTcThreads) {
            const int row = r0 + e / (NV / 4), c = (e % (NV / 4)) * 4;
            const int m = rb * kTcRows + row;
            if (m >= p.M || col0 + c >= p.N) continue;      // N is a multiple of 4
            const uint32_t at = area + (uint32_t)((row * kTcPartPitch + c) * 4);
            float4 v[kTcMaxSplits];
#pragma unroll
            for (int q = 0; q < kTcMaxSplits; ++q)
                if (q < p.nks) v[q] = ld_cluster_f4(cluster_map(at, (uint32_t)q));
            float4 a = v[0];
#pragma unroll
            for (int q = 1; q < kTcMaxSplits; ++q)
                if (q < p.nks) { a.x += v[q].x; a.y += v[q].y; a.z += v[q].z; a.w += v[q].w; }
            for (int q = 0; q < 3 && p.z[q] != nullptr; ++q) {
                __nv_bfloat162 h01 = __floats2bfloat162_rn(a.x, a.y), h23 = __floats2bfloat162_rn(a.z, a.w);
                *reinterpret_cast<uint2*>(p.z[q] + (size_t)m * p.z_pitch + col0 + c) = make_uint2(*reinterpret_cast<uint32_t*>(&h01), *reinterpret_cast<uint32_t*>(&h23));
                a.x -= __low2float(h01); a.y -= __high2float(h01); a.z -= __low2float(h23); a.w -= __high2float(h23);
            }
        }
        if (p.nks > 1) cluster_sync_exec();       // the others have read this CTA's tile
    }
}

// ------------------------------------------------------------------------------------------
// Merge the P per-slab records of each row.  Two rows per CTA, two warps per row: one takes the
// row's log-sum-exp, the other its k best entries (bound from the records' first entries, the few
// entries above it ordered by counting).
__global__ void __launch_bounds__(128) k_tc_merge(const float* __restrict__ part, int M, int P, int k,
                                                  int32_t* __restrict__ ids, float* __restrict__ logprobs)
{
    __shared__ float lse_s[2];
    __shared__ unsigned long long out_s[2][kMaxK];
    __shared__ __align__(16) unsigned char area_s[4][kMergeWarpBytes];
    pdl_launch_dependents();     // the first kernel of the next call may come up behind this one
    pdl_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r2 = warp >> 1, row = blockIdx.x * 2 + r2;
    if (row < M) {
        if (P <= 5 * 32) merge_task<5>(part, P, k, row, warp & 1, lane, &lse_s[r2], out_s[r2], area_s[warp]);
        else merge_task<kMergeLists>(part, P, k, row, warp & 1, lane, &lse_s[r2], out_s[r2], area_s[warp]);
    }
    __syncthreads();
    if ((warp & 1) == 0 && row < M && lane < k) {
        ids[(size_t)row * k + lane] = cand_id(out_s[r2][lane]);
        logprobs[(size_t)row * k + lane] = key2f(cand_key(out_s[r2][lane])) - lse_s[r2];
    }
}

// ------------------------------------------------------------------------------------------
// Shapes the head kernel takes; X = z comes in this library's own scratch, X = h straight from the caller.
bool tensor_ok(int M, bool lowrank, int K, int N, int k, int mode)
{
    if (M < 1 || K < kTcKChunk || (!lowrank && K % 8 != 0) || N % 8 != 0 || N < 64) return false;
    if (mode == 0 && (k < 1 || k > kTcMaxK)) return false;
    return true;
}

bool tensor_code_ok(int d, int r) { return d >= kTcKChunk && d % 8 == 0 && r >= kTcKChunk && r % 8 == 0; }

static constexpr size_t kTcSmemMax = 227 * 1024 - 512;   // dynamic shared memory per CTA (a little static on top)

// Merge kernel: P split-V records per row -> ids / log-probs; launched early behind the kernel that writes them.
cudaError_t merge_records(const float* part, int M, int P, int k, int32_t* ids, float* logprobs, cudaStream_t st)
{
    return launch_chain(k_tc_merge, (M + 1) / 2, 128, 0, true, st, part, M, P, k, ids, logprobs);
}

// Chooses the ring depth (and whether X can stay resident) and launches.
template <int CG, int NV>
static cudaError_t launch_gemm(TcParams p, int grid, bool pdl, cudaStream_t st)
{
    const size_t x_bytes = (size_t)p.xbox_bytes * (p.split ? 2 : 1), w_bytes = (size_t)kTcKChunk * (NV / CG) * 2;
    const size_t x_all = (size_t)((p.chunks + p.nks - 1) / p.nks) * x_bytes;
    p.xres = (p.mode != 2 && p.chunks <= kTcMaxResident && x_all + 4 * w_bytes + 1024 <= kTcSmemMax) ? 1 : 0;
    const size_t stage = w_bytes + (p.xres ? 0 : x_bytes);
    // The MMA reads 128 rows of X, also where a box has fewer; behind the last stage's X there has to be shared memory for that.
    // (Behind a resident X there is the ring: four stages of 8 KB at least.)
    const size_t read_to = (size_t)kTcRows * 128 + (p.split ? (size_t)p.xbox_bytes : 0);
    const size_t over = !p.xres && read_to > stage ? read_to - stage : 0;
    const size_t fixed = 1024 + (p.xres ? x_all : 0) + over;
    int ns = (int)((kTcSmemMax - fixed) / stage);
    if (ns > kTcMaxStages) ns = kTcMaxStages;
    if (ns < 2) return cudaErrorInvalidValue;
    p.ns = ns;
    size_t smem = fixed + (size_t)ns * stage;
    if (p.mode == 0 && smem < 1024 + kTcSortBytes) smem = 1024 + kTcSortBytes;      // room for the final sort of the lists
    if (p.mode == 2 && smem < 1024 + (size_t)kTcRows * kTcPartPitch * 4) smem = 1024 + (size_t)kTcRows * kTcPartPitch * 4;
    return launch_chain_cluster(k_tc_gemm<CG, NV>, grid, CG == 2 ? 2 : p.nks, kTcThreads, smem, pdl, st, p);
}

cudaError_t tensor_prepare(int (&max_clusters)[kTcMaxSplits + 1])
{
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_tc_gemm<1, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemMax)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_tc_gemm<1, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemMax)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_tc_gemm<2, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemMax)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_tc_gemm<1, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemMax)) != cudaSuccess) return e;
    max_clusters[0] = max_clusters[1] = 1 << 30;
    for (int c = 2; c <= kTcMaxSplits; ++c) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kTcThreads);
        cfg.dynamicSmemBytes = kTcSmemMax;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)c;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        if ((e = cudaOccupancyMaxActiveClusters(&max_clusters[c], k_tc_gemm<1, 128>, &cfg)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

struct TcShape {
    int cg, nv, nrb, nct, gct;       // CTAs a tile, its columns, row blocks (of 128 cg rows), column tiles, CTAs (pairs) per row block
};
static TcShape tc_shape(int M, int N, int sm_count)
{
    TcShape g;
    g.cg = M > kTcRows ? 2 : 1;
    g.nv = 256;
    const int rows = kTcRows * g.cg;
    g.nrb = (M + rows - 1) / rows;
    g.nct = (N + g.nv - 1) / g.nv;
    g.gct = sm_count / g.cg / g.nrb;
    if (g.gct < 1) g.gct = 1;
    if (g.gct > g.nct) g.gct = g.nct;
    if (g.gct > kMaxRecords / 2) g.gct = kMaxRecords / 2;       // the merge takes up to 320 lists per row
    return g;
}

// Does the context's scratch hold the split-V records of this call?
bool tensor_records_fit(int M, int N, int k, const Scratch& s, int sm_count)
{
    return (size_t)M * 2 * rec_row_pairs(2 * tc_shape(M, N, sm_count).gct, k) <= s.part_elems;
}

// out = X W through the tensor cores.  mode 0: top-k records then merge into ids / logprobs;
// mode 1: fp32 logits.  X is bf16 [M][K], rows x_pitch elements apart, W bf16 [K][N].
cudaError_t tensor_head(const bf16* X, const bf16* Xlo, int x_pitch, const bf16* W, int M, int K, int N, int k, int mode, int32_t* ids,
                        float* logprobs, float* logits, const Scratch& s, unsigned int epoch, int sm_count, int* launches,
                        cudaEvent_t ev0, cudaEvent_t ev1, cudaStream_t st)
{
    TcParams p;
    memset(&p, 0, sizeof(p));
    const TcShape g = tc_shape(M, N, sm_count);
    // a single row block loads only as many rows of X as there are (in whole groups of eight)
    const int xrows = M >= kTcRows ? kTcRows : (M + 7) / 8 * 8;
    if (!make_map_pitched(&p.mapX, X, M, K, x_pitch, kTcKChunk, xrows) || !make_map(&p.mapW, W, K, N, 64, kTcKChunk))
        return cudaErrorInvalidValue;
    if (Xlo != nullptr) {
        if (!make_map_pitched(&p.mapX2, Xlo, M, K, x_pitch, kTcKChunk, xrows)) return cudaErrorInvalidValue;
        p.split = 1;
    }
    p.xbox_bytes = xrows * kTcKChunk * 2;
    p.M = M; p.N = N;
    p.nrb = g.nrb; p.nct = g.nct; p.gct = g.gct;
    p.nks = 1;
    p.chunks = (K + kTcKChunk - 1) / kTcKChunk;
    p.mode = mode;
    p.k = k;
    p.out = logits;
    p.part = s.part;
    p.bound = s.bound;
    p.bound_pitch = s.bound_pitch;
    p.epoch = epoch;
    p.err = s.err;
    if (mode == 0 && (size_t)M * 2 * rec_row_pairs(2 * p.gct, k) > s.part_elems) return cudaErrorInvalidValue;
    cudaError_t e;
    const int grid = p.gct * p.nrb * g.cg;
    // optional events directly around the kernel that streams the weights (they also keep it from
    // overlapping its neighbours)
    if (ev0 && (e = cudaEventRecord(ev0, st)) != cudaSuccess) return e;
    e = g.cg == 2 ? launch_gemm<2, 256>(p, grid, !ev0, st) : launch_gemm<1, 256>(p, grid, !ev0, st);
    if (e != cudaSuccess) return e;
    if (ev1 && (e = cudaEventRecord(ev1, st)) != cudaSuccess) return e;
    *launches += 1;
    if (mode == 0) {
        e = merge_records(s.part, M, 2 * p.gct, k, ids, logprobs, st);
        *launches += 1;
    }
    return e;
}

// z = h A through the tensor cores, as up to three bf16 matrices [M][z_pitch]: the K of a tile of 128
// rows is split over the CTAs of a cluster, which add their partial tiles through distributed shared memory.
cudaError_t tensor_downproj(const bf16* h, const bf16* A, int M, int d, int r, bf16* const (&z)[3], int z_pitch, const Scratch& s,
                            int sm_count, int* launches, cudaStream_t st)
{
    TcParams p;
    memset(&p, 0, sizeof(p));
    const int xrows = M >= kTcRows ? kTcRows : (M + 7) / 8 * 8;
    if (!make_map(&p.mapX, h, M, d, kTcKChunk, xrows) || !make_map(&p.mapW, A, d, r, 64, kTcKChunk))
        return cudaErrorInvalidValue;
    p.xbox_bytes = xrows * kTcKChunk * 2;
    p.M = M; p.N = r;
    p.nrb = (M + kTcRows - 1) / kTcRows;
    // Tiles of 64 columns while clusters of four of them fit: half as much to add up per CTA (128 rows, d = 4096, r = 512, whole
    // call: 51.3 us with tiles of 128 columns, 46.8 with 64; 64 rows 46.0 / 43.3, 512 rows 74.9 / 74.4).
    const bool narrow = p.nrb * ((r + 63) / 64) <= s.max_clusters[4];
    p.nct = narrow ? (r + 63) / 64 : (r + 127) / 128;
    p.chunks = (d + kTcKChunk - 1) / kTcKChunk;
    // As many K splits as one wave of clusters takes (fewer clusters fit than SMs suggest: 15 of eight CTAs with this much
    // shared memory, 33 of four; 512 rows, d = 4096, r = 512, 16 tiles: 22.6 us with eight splits, two waves, 12 us with four).
    int nks = p.chunks < kTcMaxSplits ? p.chunks : kTcMaxSplits;
    while (nks > 1 && p.nrb * p.nct > s.max_clusters[nks]) --nks;
    p.nks = nks;
    p.gct = p.nct;
    p.mode = 2;
    p.k = 1;
    for (int q = 0; q < 3; ++q) p.z[q] = z[q];
    p.z_pitch = z_pitch;
    p.err = s.err;
    // Launched early even as the first kernel of a call: apart from the weights it touches global memory only after its
    // griddepcontrol.wait, so it may come up under the tail of whatever kernel precedes it.
    *launches += 1;
    return narrow ? launch_gemm<1, 64>(p, p.nrb * p.nct * nks, true, st) : launch_gemm<1, 128>(p, p.nrb * p.nct * nks, true, st);
}

}  // namespace slimspec
