// Streaming path for three to 64 rows: the K x V weight matrix is read from HBM exactly once, in split-V
// slabs (one CTA per SM), and multiplied on the tcgen05 tensor cores with the vocabulary on the 128-row
// side of the instruction and the batch on its N side.
//
//   D[vocabulary id][row] = W^T z^T:   A operand = weights, straight from their row-major layout (MN-major),
//                                      B operand = the code z, row-major (K-major), D in tensor memory.
//
// What bounds it: HBM.  The order of the stream is what decides how much of HBM it gets: a stage is 32 rows of
// K times the WHOLE width of the slab (14 boxes of 64 columns for a 128K vocabulary), so that an SM asks for
// 1.8 KB of consecutive bytes per row at a time.  A bare ring of that shape read 7.1 TB/s here, rings that walk
// one 128-column tile after another through all of K 6.0 to 6.2 TB/s, the same ring with slabs that do not
// start on a 128-byte line 5.8 TB/s, boxes of 16 rows 6.0 TB/s (bound by the issue of the TMA
// instructions, about 50 ns each as one lane issued them then), four stages in flight 6.8 TB/s against 7.1 TB/s with two.
// So all tiles of the slab keep their accumulators in tensor memory until the stream has ended: 7 tiles x 64
// columns for 64 rows and a 128K vocabulary.  z travels with the stages (each 32-column piece is used once).
// The tensor pipe is idle most of the time: a 128 x N x 16 instruction takes about 32 cycles up to N = 64
// (bound by the weights' way out of shared memory), 448 to 896 cycles a stage where HBM needs 2200.
//
// Precision: z is carried as two bf16 parts (value and rounding remainder), exact to about 2^-17.  Where
// tensor memory has room the parts are stacked on the N side (one instruction, two sets of columns,
// added when the logits are read), else they are two instructions into the same accumulator.
//
// Matrices that TMA does not take (a vocabulary that is no multiple of 8, unaligned pointers) come in through registers:
// warps 2..15 read the aligned 16-byte words around each piece, shift, and store it where TMA would
// have put it (RAGGED).  The code then has three parts, which is all of fp32.
//
// After the stream the logits go row group by row group through shared memory (the ring is idle then), a warp
// takes a row (maximum, bound below the row's k-th best, sum of exp, candidates, record) and the last CTAs to
// arrive merge the records (Section 4.1, up-projection; the softmax of Section 3.2; the candidate selection).
#include "kernels.h"
#include "ptx.cuh"
#include "select.cuh"
#include "epilogue.cuh"
#include "tmap.h"
#include <float.h>
#include <string.h>

namespace slimspec {

static constexpr int kSlabThreads = 512;             // warp 0 loads, warp 1 issues the MMAs; all sixteen share the tail
static constexpr int kSlabStageK = 32;               // rows of the matrix per stage
static constexpr int kSlabBox = kSlabStageK * 128;   // bytes of one box: 32 rows x 64 columns
static constexpr int kSlabMaxTiles = 14;             // most 128-column tiles a slab may have
static constexpr int kSlabMaxStages = 8;
static constexpr size_t kSlabRingBytes = 120 * 1024; // the ring stops growing here: more in flight made HBM slower, not faster
static constexpr size_t kSlabSmemMax = 226 * 1024;

struct alignas(64) SlabParams {
    CUtensorMap mapW;      // W[K][V]: box 64 columns x 32 rows, 128-byte swizzle
    CUtensorMap mapZ;      // code (high part) [M][K]: box 32 columns x zrows rows, 64-byte swizzle
    CUtensorMap mapZ2;     // its remainder, same shape
    CUtensorMap mapZ3;     // what the two leave
    const bf16* W;         // ragged: the matrix [K][V]
    int K;
    int M, V, k, mode;
    int ncta;              // slabs
    int unit_cols, units_base, units_rem;    // slab c has units_base + (c < units_rem) units of unit_cols columns
    int nst, ns;           // stages of the call, stages of the ring
    int parts, stacked;    // parts the code comes in (1..3); 1: stacked on the N side of one instruction
    int zrows;             // rows of one part in shared memory
    int tcols;             // columns of tensor memory per tile (N of the instruction)
    int tmem_cols;         // columns allocated
    int stage_bytes, wstage_bytes;
    int raw_off;           // ragged: where the feeders' slots begin, past the ring
    int lpitch;            // floats between two rows of logits in shared memory
    unsigned int idesc;
    int32_t* ids;
    float* logprobs;
    float* logits;
    float* part;
    unsigned int* ticket;
    unsigned int ticket_base;
    int* err;
};

// One row of the slab, by one warp, from its logits in shared memory (nj x 128 of them, -FLT_MAX past ncols): maximum,
// sum of exp, k best (key, id) pairs, written as the slab's record.  The k-th largest of the lanes' maxima (of
// 32 groups of columns up to k = 12, 64 up to 32, 128 beyond) bounds the row's k-th best from below; the logits
// that reach it are marked in a bit mask, parked and ordered by counting.  What counts here is the number of
// instructions and of divergent branches: a version that kept a lane's 56 columns in registers with all loops
// unrolled took 7900 cycles a row, one that parked candidates as it met them (shared-memory atomics) 5400.
// area: kSlabRowBytes of shared memory of this warp, 16-byte aligned.
static constexpr int kSlabRowBytes = (kCand + 4) * 8;
__device__ __forceinline__ void slab_row_record(const float* lr, int nj, int ncols, int col_base, int k, float* part, int row, int P, unsigned char* area, int lane)
{
    auto rec = [&](int u) -> float2& { return *rec_pair(part, row, P, k, blockIdx.x, u); };
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(area);
    const float4* lr4 = reinterpret_cast<const float4*>(lr) + lane;
    float m4[4] = {-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
#pragma unroll 2
    for (int j = 0; j < nj; ++j) {
        const float4 v = lr4[j * 32];
        m4[0] = fmaxf(m4[0], v.x);
        m4[1] = fmaxf(m4[1], v.y);
        m4[2] = fmaxf(m4[2], v.z);
        m4[3] = fmaxf(m4[3], v.w);
    }
    const float lm = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
    uint32_t kb;
    if (k <= 12) {
        kb = warp_kth_rounds(f2key(lm), k);
    } else if (k <= 32) {
        const uint32_t key[2] = {f2key(fmaxf(m4[0], m4[1])), f2key(fmaxf(m4[2], m4[3]))};
        kb = warp_kth_bisect<2>(key, k);
    } else {
        const uint32_t key[4] = {f2key(m4[0]), f2key(m4[1]), f2key(m4[2]), f2key(m4[3])};
        kb = warp_kth_bisect<4>(key, k);
    }
    const float cm = warp_max(lm);
    // (Where fewer than k groups hold columns, in a narrow slab, the bound is -FLT_MAX: every column is then a candidate.)
    const float thr = fmaxf(key2f(kb), -FLT_MAX);
    float s = 0.f;
    unsigned long long hits = 0ull;          // bit 4 j + e: column 128 j + 4 lane + e reaches the bound
#pragma unroll 2
    for (int j = 0; j < nj; ++j) {
        const float4 v = lr4[j * 32];
        s += (__expf(v.x - cm) + __expf(v.y - cm)) + (__expf(v.z - cm) + __expf(v.w - cm));
        const uint32_t nib = (v.x >= thr ? 1u : 0u) | (v.y >= thr ? 2u : 0u) | (v.z >= thr ? 4u : 0u) | (v.w >= thr ? 8u : 0u);
        hits |= (unsigned long long)nib << (4 * j);
    }
    s = warp_sum(s);
    if (lane == 0) rec(0) = make_float2(cm, s);
    int n, pos = warp_exclusive_sum(__popcll(hits), lane, &n);
    if (n <= kCand) {
        while (hits != 0ull) {
            const int b = __ffsll((long long)hits) - 1;
            hits &= hits - 1ull;
            const int c = (b >> 2) * 128 + lane * 4 + (b & 3);
            const float x = lr[c];
            if (c < ncols) cand[pos] = cand_word(f2key(x), col_base + c);
            else cand[pos] = 0ull;          // only where the bound is -FLT_MAX: no candidate
            ++pos;
        }
    }
    __syncwarp();
    if (n <= kCand) {
        warp_rank_words(cand, n, k, lane, [&](int rank, unsigned long long c) {
            rec(1 + rank) = make_float2(__uint_as_float(cand_key(c)), __int_as_float(cand_id(c)));
        });
        for (int j = n + lane; j < k; j += 32) rec(1 + j) = make_float2(__uint_as_float(0u), __int_as_float(kNoId));
    } else {
        // masses of equal logits: k rounds over the row, each taking the best logit after the previous winner
        uint32_t lk = 0xffffffffu;
        int li = -1;
        for (int j = 0; j < k; ++j) {
            uint32_t bk = 0u;
            int bi = kNoId;
            for (int c = lane; c < ncols; c += 32) {
                const uint32_t ke = f2key(lr[c]);
                const int ie = col_base + c;
                if (after(ke, ie, lk, li) && better(ke, ie, bk, bi)) { bk = ke; bi = ie; }
            }
            const uint32_t wk = warp_max_u32(bk);
            const uint32_t wi = warp_min_u32(bk == wk ? (uint32_t)bi : 0xffffffffu);
            lk = wk;
            li = (int)wi;
            if (lane == 0) rec(1 + j) = make_float2(__uint_as_float(wk), __int_as_float(wk != 0u ? (int)wi : kNoId));
            if (wk == 0u) { lk = 0u; li = kNoId; }
        }
    }
    __syncwarp();
}

// Weights through registers (RAGGED).  Rows eight apart are equally far off a 16-byte boundary, whatever V is, so the
// shift is dealt out by warp: one of the sixteen feeders has a row below 16 and the one 16 further on of every
// stage and runs one of four loops, each with its shift in words built in.  A step of the loop is 31 pieces of
// 16 bytes (8 columns) of both rows: the 32 aligned words that cover them come in by cp.async, a word a lane,
// kSlabSteps steps in flight, each in a slot of its own; then the warp shifts them and stores them where TMA would
// have.  What counts is the number of instructions (about 20 for 496 bytes; with rows dealt to warps in turn, shift
// and bounds worked out for each, it was 150, 74 % of the issue slots were busy and the stream ran at 1.0 to 2.0 TB/s)
// and of loops: with eight, one for each shift in elements, the warps starved for instructions at 0.7 TB/s.
static constexpr int kSlabSteps = 4;
static constexpr int kSlabFeeders = 16;
struct SlabFeed {
    const bf16* W;
    int V, K, col0, nu, nst, ns;         // nu: pieces of a row
    int row0;                            // the warp's first row of a stage; the other is 16 further on
    uint32_t raw, ring;                  // the lane's word of the warp's first slot; the ring (shared-memory addresses)
    int stage_bytes;
    uint64_t *full, *empty;
    volatile int* abort_flag;
    int* err;
};

// The lane's word at q where it need not lie inside the matrix, [beg, end): zeros elsewhere.
__device__ __noinline__ void slab_feed_edge(uint32_t dst, const char* q, const char* beg, const char* end)
{
    if (q >= beg && q + 16 <= end) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(q) : "memory");
        return;
    }
    for (int t = 0; t < 16; t += 2) {
        const unsigned short w = q + t >= beg && q + t < end ? *reinterpret_cast<const unsigned short*>(q + t) : (unsigned short)0;
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(dst + t), "h"(w) : "memory");
    }
}

template <int WORDS>
__device__ __forceinline__ void slab_feed(const SlabFeed& f, uint32_t sh)
{
    const int lane = threadIdx.x & 31;
    const int runs = (f.nu + 30) / 31;
    const char* beg = reinterpret_cast<const char*>(f.W);
    const char* end = beg + (size_t)f.K * f.V * sizeof(bf16);
    const long long pitch = 2ll * f.V;
    const long long down16 = 16 * pitch;
    const char* q = beg + 2 * (size_t)f.col0 + f.row0 * pitch - 2 * (int)sh + 16 * lane;       // next word to send for, of the first row
    int qu = 0, qi = 0;
    auto send = [&](uint32_t dst) {
        if (qi < f.nst) {
            if (qi > 0 && (qi + 1) * kSlabStageK < f.K && f.V >= 256) {          // a row away from the matrix's ends
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n\tcp.async.cg.shared.global [%2], [%3], 16;" ::"r"(dst), "l"(q),
                             "r"(dst + 512), "l"(q + down16)
                             : "memory");
            } else {
                slab_feed_edge(dst, q, beg, end);
                slab_feed_edge(dst + 512, q + down16, beg, end);
            }
            q += 496;
            if (++qu == runs) { qu = 0; ++qi; q += 2 * down16 - 496 * runs; }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int d = 0; d < kSlabSteps; ++d) send(f.raw + d * 1024);
    int s = 0, ph = 0, slot = 0;
    const uint32_t bits = (sh & 1u) * 16u;
    const uint32_t x0 = (uint32_t)(f.row0 * 128);            // both rows have the same place modulo 8
    for (int i = 0; i < f.nst; ++i) {
        if (i >= f.ns && !mbar_wait_warp(&f.empty[s], ph ^ 1, f.abort_flag, f.err, ERR_WAIT_EMPTY)) break;
        const uint32_t stage = f.ring + (uint32_t)(s * f.stage_bytes) + x0;
        for (int u = 0, piece = lane; u < runs; ++u, piece += 31) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kSlabSteps - 1) : "memory");
            __syncwarp();
            const uint32_t src = f.raw + slot * 1024, other = lane < 31 ? 16u : 0u;
            uint4 a[2], b[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                a[h] = lds128(src + h * 512);
                b[h] = lds128(src + h * 512 + other);
            }
            const uint32_t dst = stage + (uint32_t)((piece >> 3) * kSlabBox + (((piece ^ f.row0) & 7) << 4));
            if (lane < 31 && piece < f.nu) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t w[8] = {a[h].x, a[h].y, a[h].z, a[h].w, b[h].x, b[h].y, b[h].z, b[h].w};
                    uint32_t o[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) o[j] = __funnelshift_r(w[j + WORDS], w[j + WORDS + 1], bits);
                    sts128(dst + h * 2048, o[0], o[1], o[2], o[3]);
                }
            }
            __syncwarp();                                    // everyone has read the slot
            send(src);
            slot = (slot + 1) % kSlabSteps;
        }
        fence_proxy_async_shared();
        __syncwarp();
        if (lane == 0) mbar_arrive(&f.full[s]);
        if (++s == f.ns) { s = 0; ph ^= 1; }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// RG: rows the tail takes at a time (8, 16 or 32).  At most 112 registers, so that a CTA of the next call's
// down-projection (128 threads) finds room beside this one.
static constexpr int kSlabRaggedThreads = kSlabThreads + 64;      // RAGGED: two warps more, so that sixteen feed; the tail is the first sixteen's
template <int RG, bool RAGGED>
__global__ void __maxnreg__(RAGGED ? 96 : 112) k_slab_head(const __grid_constant__ SlabParams p)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t full[kSlabMaxStages], empty[kSlabMaxStages], acc_full;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ unsigned int ticket_s;
    unsigned char* ring = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    volatile int* abort_flag = &abort_s;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;      // the same in all lanes, for the compiler too
    const int cta = blockIdx.x;
    const int my_units = p.units_base + (cta < p.units_rem ? 1 : 0);
    const int col0 = (cta * p.units_base + min(cta, p.units_rem)) * p.unit_cols;
    const int ncols = min(my_units * p.unit_cols, p.V - col0);
    const int nbox = (ncols + 63) >> 6, ntile = (nbox + 1) >> 1;

    if (tid == 0) {
        for (int s = 0; s < kSlabMaxStages; ++s) { mbar_init(&full[s], RAGGED ? 1 + kSlabFeeders : 1); mbar_init(&empty[s], 1); }
        mbar_init(&acc_full, 1);
        abort_s = 0;
        mbar_fence_init();
        if (!RAGGED) prefetch_tensor_map(&p.mapW);
        prefetch_tensor_map(&p.mapZ);
        if (p.parts >= 2) prefetch_tensor_map(&p.mapZ2);
    }
    if (warp == 1) tmem_alloc(&tmem_base_s, (uint32_t)p.tmem_cols);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);

    if (warp == 0) {
        // ================= producer.  The weights are final before the call is made (the contract of the
        // library), so the first stages' weights are sent for before the kernel ahead has finished; the
        // code comes from that kernel.
        const uint32_t zpart = (uint32_t)p.zrows * 64u;
        const uint32_t bytes = (RAGGED ? 0u : (uint32_t)nbox * kSlabBox) + zpart * (uint32_t)p.parts;
        const int npre = min(p.ns, p.nst);
        auto send_w = [&](int i, int s) {
            unsigned char* dst = ring + (size_t)s * p.stage_bytes;
            mbar_arrive_expect_tx(&full[s], bytes);
            if (!RAGGED)
                for (int b = 0; b < nbox; ++b) tma_load_2d(dst + b * kSlabBox, &p.mapW, col0 + b * 64, i * kSlabStageK, &full[s]);
        };
        auto send_z = [&](int i, int s) {
            unsigned char* dst = ring + (size_t)s * p.stage_bytes + p.wstage_bytes;
            tma_load_2d(dst, &p.mapZ, i * kSlabStageK, 0, &full[s]);
            if (p.parts >= 2) tma_load_2d(dst + zpart, &p.mapZ2, i * kSlabStageK, 0, &full[s]);
            if (p.parts == 3) tma_load_2d(dst + 2 * zpart, &p.mapZ3, i * kSlabStageK, 0, &full[s]);
        };
        if (elect_one())
            for (int i = 0; i < npre; ++i) send_w(i, i);
        __syncwarp();
        pdl_launch_dependents();
        pdl_wait();
        if (elect_one())
            for (int i = 0; i < npre; ++i) send_z(i, i);
        __syncwarp();
        int s = 0, ph = 0;
        bool alive = true;
        for (int i = npre; i < p.nst; ++i) {
            if (alive) alive = mbar_wait_uniform(&empty[s], ph);
            if (alive) {
                if (elect_one()) {
                    send_w(i, s);
                    send_z(i, s);
                }
                __syncwarp();
            }
            if (++s == p.ns) { s = 0; ph ^= 1; }
        }
        if (!alive) mbar_gave_up(abort_flag, p.err, ERR_WAIT_EMPTY);
    } else if (warp == 1) {
        // ================= MMA issuer: per stage two steps of 16 along K for every tile.  All tiles get one part of the code
        // before any gets the next: two instructions in a row into the same accumulator wait for one another (64 rows,
        // d = 8192, r = 1024: 115 us part by part in each tile, 86 us this way).
        // The warp runs the loop together and elects a lane at each issue (see mbar_wait_uniform).
        constexpr uint32_t A_HI = (1024u >> 4) | (1u << 14) | (2u << 29);      // SBO: 8 rows of K; version 1; 128-byte swizzle
        constexpr uint32_t B_HI = (512u >> 4) | (1u << 14) | (4u << 29);       // SBO: 8 rows of z; 64-byte swizzle
        const uint32_t ring_w = (smem_u32(ring) >> 4) & 0x3fffu;
        const uint32_t a_lbo = (uint32_t)(kSlabBox >> 4) << 16;                // LBO: the tile's second 64 columns
        const uint32_t stage_w = (uint32_t)p.stage_bytes >> 4, z_off = (uint32_t)p.wstage_bytes >> 4;
        const uint32_t z_part = (uint32_t)(p.zrows * 64) >> 4;
        const int passes = p.stacked ? 1 : p.parts;
        int s = 0, ph = 0;
        uint32_t st = ring_w;
        bool alive = true;
        pdl_wait();          // nothing to do before the code is there, and the waits below are bounded
        for (int i = 0; i < p.nst; ++i) {
            if (alive) alive = mbar_wait_uniform(&full[s], ph);
            if (alive) {
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk) {
                        for (int q = 0; q < passes; ++q) {
                            uint32_t a = (st + (uint32_t)(kk * 128)) | a_lbo, d = tmem_base;
                            const uint32_t b = (st + z_off + (uint32_t)(kk * 2) + (uint32_t)q * z_part) | (1u << 16);
                            const uint32_t acc = (i | kk | q) ? 1u : 0u;
                            for (int t = 0; t < ntile; ++t) {
                                tc_mma_bf16_words2(d, a, A_HI, b, B_HI, p.idesc, acc);
                                a += (uint32_t)(2 * kSlabBox) >> 4;
                                d += (uint32_t)p.tcols;
                            }
                        }
                    }
                    tc_commit(&empty[s]);
                    if (i == p.nst - 1) tc_commit(&acc_full);
                }
                __syncwarp();
            }
            st += stage_w;
            if (++s == p.ns) { s = 0; ph ^= 1; st = ring_w; }
        }
        if (!alive) mbar_gave_up(abort_flag, p.err, ERR_WAIT_FULL);
    } else if (RAGGED) {
        // ================= feeders
        SlabFeed f;
        f.W = p.W; f.V = p.V; f.K = p.K; f.col0 = col0; f.nu = (ncols + 7) >> 3; f.nst = p.nst; f.ns = p.ns;
        // Of an odd V the rows' shifts run through all eight values: the four feeders of a scheduler get two shifts that share
        // a loop (two loops on one scheduler do not fit its instruction buffer: 147 us instead of 95 us for
        // d = 3072, V = 50257).  Of an even V rows four apart have the same shift, and the plain order does that.
        if (p.V & 1) {
            const int n = (warp - 2) >> 2, sh0 = (int)(reinterpret_cast<uintptr_t>(p.W + col0) & 15) >> 1;
            f.row0 = (((2 * (warp & 3) + (n & 1) - sh0) * p.V) & 7) + 8 * (n >> 1);        // an odd number is its own inverse modulo 8
        } else {
            f.row0 = ((warp - 2) & 7) + 8 * ((warp - 2) >> 3);
        }
        f.ring = smem_u32(ring);
        f.raw = f.ring + p.raw_off + (warp - 2) * (kSlabSteps * 1024) + lane * 16;
        f.stage_bytes = p.stage_bytes;
        f.full = full; f.empty = empty; f.abort_flag = abort_flag; f.err = p.err;
        const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(p.W + (size_t)f.row0 * p.V + col0) & 15) >> 1;
        switch (sh >> 1) {
        case 0: slab_feed<0>(f, sh); break;
        case 1: slab_feed<1>(f, sh); break;
        case 2: slab_feed<2>(f, sh); break;
        default: slab_feed<3>(f, sh); break;
        }
    }

    // ================= tail: all warps.  Everything below writes what belongs to the kernels ahead in the stream.
    pdl_wait();          // before the bounded wait: what the kernels ahead take is not this one's
    const bool ok = mbar_wait_warp(&acc_full, 0, abort_flag, p.err, ERR_WAIT_ACC);
    tc_fence_after_sync();
    float* lg = reinterpret_cast<float*>(ring);          // the ring is idle: every stage has been multiplied
    unsigned char* row_area = reinterpret_cast<unsigned char*>(lg + (size_t)RG * p.lpitch) + warp * kSlabRowBytes;
    const int q = warp & 3;                              // the lane quarter of tensor memory this warp may read
    for (int r0 = 0; ok && r0 < p.M; r0 += RG) {
        if (r0 > 0) __syncthreads();                     // the rows before have been worked off
        for (int t = warp >> 2; t < ntile && warp < kSlabThreads / 32; t += kSlabThreads / 128) {
            const uint32_t ta = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(t * p.tcols + r0);
            uint32_t v[RG];
            tmem_ld(ta, v);
            tmem_ld_wait();
            if (p.stacked) {
#pragma unroll 1
                for (int part = 1; part < p.parts; ++part) {
                    uint32_t w[RG];
                    tmem_ld(ta + (uint32_t)(part * p.zrows), w);
                    tmem_ld_wait();
#pragma unroll
                    for (int n = 0; n < RG; ++n) v[n] = __float_as_uint(__uint_as_float(v[n]) + __uint_as_float(w[n]));
                }
            }
            const int c = t * 128 + q * 32 + lane;
            if (p.mode == 0) {
#pragma unroll
                for (int n = 0; n < RG; ++n) lg[(size_t)n * p.lpitch + c] = c < ncols ? __uint_as_float(v[n]) + 0.f : -FLT_MAX;     // -0 becomes +0: keys and compares agree
            } else if (c < ncols) {
#pragma unroll
                for (int n = 0; n < RG; ++n)
                    if (r0 + n < p.M) p.logits[(size_t)(r0 + n) * p.V + col0 + c] = __uint_as_float(v[n]) + 0.f;
            }
        }
        if (p.mode == 0) {
            __syncthreads();
            const int rows = min(RG, p.M - r0);
            for (int n = warp; n < rows && warp < kSlabThreads / 32; n += kSlabThreads / 32) {
                const float* lr = lg + (size_t)n * p.lpitch;
                slab_row_record(lr, ntile, ncols, col0, p.k, p.part, r0 + n, p.ncta, row_area, lane);
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 1) tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    if (p.mode == 0 && abort_s == 0) merge_by_last_arrivals(p, &ticket_s, ring);
}

// ------------------------------------------------------------------------------------------
struct SlabGeometry {
    int ncta, unit_cols, units_base, units_rem, ntile, ns, rg;
    int zrows, stacked, tcols, tmem_cols, stage_bytes, wstage_bytes, raw_off, lpitch;
    size_t smem;
};

// Everything but the layout of W: M <= 64, k <= 64.
static bool slab_geometry(int M, int parts, int K, int V, int k, int sm_count, bool ragged, SlabGeometry* g)
{
    if (M < 1 || M > 64 || V < 1 || K < 1 || k < 1 || k > kMaxK) return false;
    const int warps = (ragged ? kSlabRaggedThreads : kSlabThreads) / 32;
    // Slabs start on a 128-byte line while that costs little balance; narrow slabs (small vocabularies)
    // are cut finer.
    int uc = 64;
    while (uc > 8 && (V + uc - 1) / uc < 4 * sm_count) uc >>= 1;
    const int units = (V + uc - 1) / uc;
    g->unit_cols = uc;
    g->ncta = units < sm_count ? units : sm_count;
    if (g->ncta > kMaxRecords) g->ncta = kMaxRecords;
    g->units_base = units / g->ncta;
    g->units_rem = units % g->ncta;
    const int cols = (g->units_base + (g->units_rem ? 1 : 0)) * uc;
    g->ntile = (cols + 127) / 128;
    if (g->ntile > kSlabMaxTiles) return false;
    g->rg = M <= 8 ? 8 : (M <= 16 || (M > 32 && M <= 48)) ? 16 : 32;      // rows of the tail's groups; 33..48 rows: three groups of 16
    const int mpad = (M + g->rg - 1) / g->rg * g->rg;
    g->zrows = parts == 2 ? mpad : (mpad < 16 ? 16 : mpad);             // N of an instruction is a multiple of 16
    g->stacked = parts > 1 && (g->ntile * parts * g->zrows <= 512 || g->zrows < 16) ? 1 : 0;
    g->tcols = g->stacked ? parts * g->zrows : g->zrows;
    if (g->ntile * g->tcols > 512) return false;
    g->tmem_cols = 32;
    while (g->tmem_cols < g->ntile * g->tcols) g->tmem_cols *= 2;
    g->wstage_bytes = g->ntile * 2 * kSlabBox;
    g->stage_bytes = g->wstage_bytes + (parts * g->zrows * 64 + 1023) / 1024 * 1024;
    int ns = (int)(kSlabRingBytes / g->stage_bytes);
    if (ns < 2) ns = 2;
    if (ns > kSlabMaxStages) ns = kSlabMaxStages;
    g->ns = ns;
    g->lpitch = g->ntile * 128;
    g->raw_off = ns * g->stage_bytes;
    size_t area = (size_t)g->raw_off + (ragged ? (size_t)kSlabFeeders * kSlabSteps * 1024 : 0);
    const size_t tail = (size_t)g->rg * g->lpitch * 4 + (size_t)(kSlabThreads / 32) * kSlabRowBytes;
    if (area < tail) area = tail;
    // the merge: R CTAs share the rows
    int R = (M + warps / 2 - 1) / (warps / 2);
    if (R > g->ncta) R = g->ncta;
    const int mine = (M + R - 1) / R;
    if (mine > 16) return false;
    if (area < (size_t)merge_area_bytes(mine, warps)) area = merge_area_bytes(mine, warps);
    g->smem = 1024 + area;
    return g->smem <= kSlabSmemMax;
}

// W as TMA takes it (rows of a multiple of 16 bytes; the pointer is the caller's to check), and the code likewise.
bool slab_ok(int M, int parts, int K, int V, int k, int sm_count)
{
    SlabGeometry g;
    return V % 8 == 0 && V >= 64 && K >= 8 && K % 8 == 0 && slab_geometry(M, parts, K, V, k, sm_count, false, &g);
}

// Any V and K, any alignment of W.
bool slab_any_ok(int M, bool lowrank, int K, int V, int k, int sm_count)
{
    SlabGeometry g;
    return slab_geometry(M, lowrank ? 3 : 1, K, V, k, sm_count, true, &g);
}

template <typename Kern>
static cudaError_t slab_allow(Kern kern) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSlabSmemMax); }

cudaError_t slab_prepare()
{
    cudaError_t e;
    if ((e = slab_allow(k_slab_head<8, false>)) != cudaSuccess || (e = slab_allow(k_slab_head<8, true>)) != cudaSuccess) return e;
    if ((e = slab_allow(k_slab_head<16, false>)) != cudaSuccess || (e = slab_allow(k_slab_head<16, true>)) != cudaSuccess) return e;
    if ((e = slab_allow(k_slab_head<32, false>)) != cudaSuccess) return e;
    return slab_allow(k_slab_head<32, true>);
}

template <int RG, bool RAGGED>
static cudaError_t slab_launch(const SlabGeometry& g, bool pdl, cudaStream_t st, const SlabParams& p)
{
    return launch_chain(k_slab_head<RG, RAGGED>, g.ncta, RAGGED ? kSlabRaggedThreads : kSlabThreads, g.smem, pdl, st, p);
}

cudaError_t slab_head(const bf16* const (&z)[3], int z_pitch, const bf16* W, int M, int K, int V, int k, int mode, int32_t* ids, float* logprobs,
                      float* logits, const Scratch& s, int sm_count, bool pdl, cudaStream_t st)
{
    SlabGeometry g;
    const int parts = z[2] != nullptr ? 3 : z[1] != nullptr ? 2 : 1;
    const bool ragged = V % 8 != 0 || V < 64 || ((uintptr_t)W & 15) != 0;
    if (!slab_geometry(M, parts, K, V, k, sm_count, ragged, &g)) return cudaErrorInvalidValue;
    SlabParams p;
    memset(&p, 0, sizeof(p));
    if (!ragged && !make_map(&p.mapW, W, K, V, 64, kSlabStageK)) return cudaErrorInvalidValue;
    CUtensorMap* mz[3] = {&p.mapZ, &p.mapZ2, &p.mapZ3};
    for (int q = 0; q < parts; ++q)
        if (!make_map_pitched(mz[q], z[q], M, K, z_pitch, 32, g.zrows)) return cudaErrorInvalidValue;
    p.W = W; p.K = K;
    p.M = M; p.V = V; p.k = k; p.mode = mode;
    p.ncta = g.ncta; p.unit_cols = g.unit_cols; p.units_base = g.units_base; p.units_rem = g.units_rem;
    p.nst = (K + kSlabStageK - 1) / kSlabStageK; p.ns = g.ns;
    p.parts = parts; p.stacked = g.stacked; p.zrows = g.zrows; p.tcols = g.tcols; p.tmem_cols = g.tmem_cols;
    p.stage_bytes = g.stage_bytes; p.wstage_bytes = g.wstage_bytes; p.raw_off = g.raw_off; p.lpitch = g.lpitch;
    // D fp32, A and B bf16, A MN-major, B K-major, N = columns of a tile, M = 128
    p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(g.tcols >> 3) << 17) | (8u << 24);
    p.ids = ids; p.logprobs = logprobs; p.logits = logits;
    p.part = s.part; p.ticket = s.tickets; p.err = s.err;
    p.ticket_base = mode == 0 ? *s.ticket_base_host : 0u;
    if (mode == 0 && (size_t)M * 2 * rec_row_pairs(p.ncta, k) > s.part_elems) return cudaErrorInvalidValue;
    const cudaError_t e = ragged ? (g.rg == 8 ? slab_launch<8, true>(g, pdl, st, p) : g.rg == 16 ? slab_launch<16, true>(g, pdl, st, p) : slab_launch<32, true>(g, pdl, st, p))
                        : g.rg == 8 ? slab_launch<8, false>(g, pdl, st, p) : g.rg == 16 ? slab_launch<16, false>(g, pdl, st, p) : slab_launch<32, false>(g, pdl, st, p);
    if (e == cudaSuccess && mode == 0) *s.ticket_base_host += (unsigned int)p.ncta;      // the tickets this launch will take
    return e;
}

}  // namespace slimspec
