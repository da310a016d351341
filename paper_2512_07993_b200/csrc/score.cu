// skipkv_score: sentence scores per (sequence, KV head) slab (paper Section 4.1).
//
//   sweeps    (one launch) pass A: log-sum-exp of every window-query row over the slab's tokens
//             (tensor cores: logits = Q_rows x K_tile^T, one thread per query row);
//             pass B: tok_imp[t] = (1/alpha) sum_w max_q 2^(s_q[w][t] - lse_q[w])   (max before exp: exp is monotone)
//             (tensor cores: logits - (lse - e) = [K_tile, 1] x [Q_block, e - lse]^T, one thread per token; e: see lse_shift);
//             in one of them the per-sentence sums of the key rows as a second product on the tile already in shared
//             memory: K_tile^T x (0/1 matrix token -> sentence slot)
//   up to 128 sentences per slab: one kernel for the rest, else
//   pool      per sentence: mean tok_imp, mean key, normalisation, split into bf16 high and low parts
//   gram x2   pairwise cosine G on the tensor cores (three bf16 products: hi.hi + hi.lo + lo.hi);
//             pass 1: Z_i = sum_{j!=i} e^{G_ij} and lam_i = max_{j>i} G_ij;
//             pass 2: red_i = (1/S) sum_{j!=i} e^{G_ij} / Z_j (G symmetric) and the final score.
//
// Logits are kept in base 2: s = (q.k) * log2(e)/sqrt(d).  |G| <= 1 so the row softmax of G
// needs no max subtraction.
//
// The sweeps are a persistent, warp-specialised kernel, one CTA per SM: a TMA warp streams 128-token key tiles (and the
// group's query rows) into shared memory, two warps issue tcgen05.mma in turn into a ring of tensor-memory accumulators,
// epilogue warpgroups take the products round-robin, and in one of the passes another warpgroup writes the 0/1
// matrices of the pooling product and reads out the pooled sums while a further warp issues
// that product.  Work is the list of 128-token tiles over all slabs cut into equal contiguous ranges, so
// ragged slabs balance.
//
// Query rows of a group are staged as blocks of WB window positions x n heads (row q*WB + w of a block), so that the n
// heads of a window position sit at a fixed column stride for the max over heads; pass A takes the same rows in
// blocks of 128.
#include <cstddef>

#include "common.cuh"
#include "tc.cuh"

namespace skipkv {

// ---------------------------------------------------------------------------------------
// Both sweeps over the keys in one persistent launch.  A CTA goes through its range of tiles twice:
//   pass A   log-sum-exp of every window-query row over the CTA's part of each slab -> one record per (CTA, slab)
//   pass B   importance of every token
// Between the two it waits, slab by slab, until every CTA that shares the slab has left its record (a counter of tiles);
// nobody waits for anything but pass A of CTAs that are all resident (one per SM), and the waits are bounded anyway.
// As two launches the second started its first tile 6 us after the first had drained.  Pass B comes back through the range, so it begins
// with the tiles that are still in shared memory (all of them where the range fits into the ring) and finds the next ones in L2.
// The per-sentence key sums are a product per tile in either pass.  With one operand of query rows (up to 128) pass A waits for DRAM, and they
// are its; with several it waits for its exponentials, wants the fourth epilogue warpgroup, and they are pass B's.  80 slabs of 16K to 32K,
// 128 rows: pass A 112 us, pass B 75 with the sums in pass A; 97 and 105 in pass B; the whole call 315 -> 294 us.  128 slabs of 32K to 64K,
// 320 rows: 757 and 425 against 606 and 490.
// What bounds the passes beside that: instructions.  A tile takes about 6000 warp instructions for 1500 exponentials' worth of work a warp, and
// the warps' different loops do not fit into the instruction caches together: a 512-instruction loop in the other warps slows
// a warp that issues products from 570 to 2800 clocks a product.  Loops are kept short, and what can be done once for several tiles is.
// ---------------------------------------------------------------------------------------
constexpr int kStagesMax = 6;
constexpr int kAccB = 3;                // pass B: accumulators of up to 160 columns, an epilogue warpgroup each
constexpr int kAccCols = 160;
constexpr int kAccAMax = 4;             // pass A: accumulators of 128 columns, an epilogue warpgroup each; three where the fourth group has the pooling
constexpr int kIndRingMax = 4;          // indicator matrices in flight (the pooled sums have two accumulators of their own)
constexpr int kIndSlots = 16;           // sentence slots of one indicator matrix
constexpr int kIndBytes = kIndSlots * 128 * 2;   // [16 slots][128 tokens] bf16 as two 64-token halves, 128-byte swizzle
constexpr uint32_t kPoolCol = kAccB * kAccCols;   // tensor-memory column of the first pooled-sum accumulator (16 columns each)
constexpr int kPoolWarps = 4;
constexpr int kSweepThreads = 20 * 32;  // TMA warp, two MMA warps, issuer of the pooling products; three epilogue warpgroups; a fourth, which has the pooling
constexpr int kExtRow = 32;             // bytes of a row of the extra K step (16 bf16)
constexpr float kLog2e = 1.4426950408889634f;

struct SweepCtl {                       // barriers and small shared state, after the tile buffers
    uint64_t full[kStagesMax], empty[kStagesMax];
    uint64_t qfull, qempty;
    // A product (of a tile and a block of query rows) goes to the accumulator of its number in the pass % accumulators; "has been read" is by
    // product number % twice the accumulators, so that each barrier has one waiter (the MMA warp whose product is the next into that
    // accumulator) that sees all its phases
    uint64_t tfull_a[kAccAMax], tempty_a[2 * kAccAMax], tfull_b[kAccB], tempty_b[2 * kAccB];
    uint64_t tokfull[4];                // pass B, several blocks per tile: the shares of a tile's tokens from all blocks but the last
    uint64_t extfull;                   // pass B: the rows' -lse as operand columns; by group that prepares them (a slab's first product's), "the
    uint64_t extempty[kAccB];           // products of the slab before have completed", so that a group sees every phase of its barrier
    // ring of indicator matrices: written by the four pooling warps -> multiplied by their issuer -> read out by the pooling warps
    uint64_t ifull[kIndRingMax], iempty[kIndRingMax];
    uint64_t pfull[2];                  // the last product of a run of tiles into accumulator i has completed
    uint64_t retired[3];                // every product of the MMA warps (0, 1) / the pooling issuer (2) has completed
    uint32_t tmem_base;
    int abort_flag;
    int ind_flags[kIndRingMax];            // 1: the tile has another matrix after this one, 2: joins the open run, 4: closes a run
    uint32_t wsum[32];
};

// Pass A, last block of at most 64 rows: on every second tile its rows take the upper tensor-memory lanes, so that the
// exponentials spread over all four schedulers.
__host__ __device__ constexpr bool sweep_can_shift(int R, int RA) { return RA > 1 && R - (RA - 1) * 128 <= 64; }
// The rows of pass B's extra K step; before, the sums of pass A: 8 bytes by warpgroup, row and block, the last block's on shifted tiles apart.
__host__ __device__ constexpr size_t sweep_ext_bytes(int R, int RA) {
    const size_t ext = size_t(RA) * 128 * kExtRow, sums = size_t(kAccAMax) * (RA + (sweep_can_shift(R, RA) ? 1 : 0)) * 128 * 8;
    return ext > sums ? ext : sums;
}

struct SweepArgs {
    int Hq, Hk, window, n_slabs, max_cap, max_sent, stages;
    int pool_a;                         // the pooling products are pass A's (1) or pass B's (0)
    int ind_log;                        // log2 of the indicator matrices in flight
    int WB, RB, N, R, RA;               // window positions per block of pass B, its blocks, their rows N = WB * n; all rows R = RB * N; blocks of pass A
    const int64_t* slab_off;
    const int32_t* cap;
    const int32_t* kv_len;
    const int32_t* sent_off;
    const int32_t* n_sent;
    float2* rec;                        // [cta + slab][RA * 128] (reference, sum) of a CTA's part of a slab
    uint32_t* lse_cnt;                  // [slabs] tiles whose records are written; zero at the start
    uint32_t* sum_cnt;                  // [slabs] four times the tiles whose key sums are stored; zero at the start
    float* tok_imp_user;
    float* tok_imp_ws;
    float* vsum;                        // [slabs][max_sent][128] sums of key rows
    uint32_t* status;
    const Header* hdr;
    const int32_t* block_table;         // nullable: paged cache, tile j of slab s is page block_table[s * max_pages + j]
    int max_pages;
    int* table;                         // [2 * n_slabs + 1] tile prefix and first cache rows, where shared memory has no room for them
};

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Bounded wait of one thread until *p reaches `want`; gives up like role_wait.  See warp_flag_wait for a whole warp.
static __device__ __noinline__ bool flag_wait(const uint32_t* p, uint32_t want, uint32_t limit, int* abort_flag, uint32_t* status) {
    for (uint32_t i = 0; i < limit; ++i) {
        if (ld_acquire(p) >= want) return true;
        if (i > 16) __nanosleep(32);
        if ((i & 255) == 255 && *reinterpret_cast<volatile int*>(abort_flag)) return false;
    }
    atomicOr(status, SKIPKV_STATUS_COPY_TIMEOUT);
    *reinterpret_cast<volatile int*>(abort_flag) = 1;
    return false;
}
// The same for a converged warp: one lane polls, and all of them see what was published.  (The vote alone orders no memory accesses; the
// barrier behind the acquire does.)
__device__ __forceinline__ bool warp_flag_wait(const uint32_t* p, uint32_t want, uint32_t limit, int* abort_flag, uint32_t* status) {
    bool ok = true;
    if ((threadIdx.x & 31) == 0) ok = flag_wait(p, want, limit, abort_flag, status);
    __syncwarp();
    return __all_sync(0xffffffffu, ok);
}

// D[128 x n] (+)= A[128 x 128] * B[n x 128]^T.  Both operands are two halves of 64 channels, a_half / b_half bytes apart.
__device__ __forceinline__ void umma_tile(uint32_t tmem_d, uint32_t a_smem, uint32_t a_half, uint32_t b_smem, uint32_t b_half, uint32_t idesc, uint32_t leader) {
    const uint64_t da = umma_desc_sw128(a_smem), db = umma_desc_sw128(b_smem);
#pragma unroll
    for (int half = 0; half < 2; ++half)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
            umma_bf16(tmem_d, da + uint64_t(half * (a_half >> 4) + ks * 2), db + uint64_t(half * (b_half >> 4) + ks * 2), idesc, (half || ks) ? 1u : 0u, leader);
}
// Descriptor of a K-major operand of 16 columns, rows 32 bytes apart, 32-byte swizzle (groups of 8 rows 256 bytes apart).
__device__ __forceinline__ uint64_t umma_desc_sw32(uint32_t smem_addr) {
    return uint64_t((smem_addr >> 4) & 0x3fffu) | (uint64_t(1) << 16) | (uint64_t(256 >> 4) << 32) | (uint64_t(1) << 46) | (uint64_t(6) << 61);
}
__device__ __forceinline__ float max3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }
// The logits of pass B are accumulated less (log-sum-exp - e), e = 1 + floor(log2 rows).  The difference lies between the row's mean
// logit - 1 and its largest one (Jensen), so the sums keep the magnitude of the logits and stay about as often positive as negative;
// the tensor core truncates when it adds.  With the whole log-sum-exp, 15 for 32K rows, they were ten times as large and all
// negative, and every importance came out 9e-7 too large.  The factor 2^-e is exact and comes with the 1 / window.
__device__ __forceinline__ int lse_shift(int rows) { return 32 - __clz(max(rows, 1)); }

// ---- pass A epilogue: one accumulator (128 tokens) folded into a row's sum of 2^(logit - m).  The reference m is the
// largest logit of the row's first 32 tokens; it stays, whatever comes later, as long as a chunk's sum is below 2^60 --
// no running maximum and no rescaling in the common case.  A chunk beyond that is folded again under a larger reference.
// `release` gives the accumulator back once its last chunk is in registers, so that the next product runs under that chunk's exponentials.
template <bool kMasked>
__device__ __forceinline__ void lse_chunk(float (&v)[32], int left, float scale, float& m, float& l) {
    if (kMasked) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j >= left) v[j] = -INFINITY;
    }
    auto chunk_max = [&]() {
        float c0 = fmaxf(v[0], v[1]), c1 = fmaxf(v[2], v[3]);
#pragma unroll
        for (int j = 4; j < 32; j += 4) { c0 = max3(c0, v[j], v[j + 1]); c1 = max3(c1, v[j + 2], v[j + 3]); }
        return fmaxf(c0, c1) * scale;
    };
    auto chunk_sum = [&]() {
        float2 s0 = make_float2(0.f, 0.f), s1 = s0;
        const float2 sc = make_float2(scale, scale), neg = make_float2(-m, -m);
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const float2 x = __ffma2_rn(make_float2(v[j], v[j + 1]), sc, neg), y = __ffma2_rn(make_float2(v[j + 2], v[j + 3]), sc, neg);
            s0 = __fadd2_rn(s0, make_float2(ex2f(x.x), ex2f(x.y)));
            s1 = __fadd2_rn(s1, make_float2(ex2f(y.x), ex2f(y.y)));
        }
        return (s0.x + s0.y) + (s1.x + s1.y);
    };
    if (m == -INFINITY) m = chunk_max();
    float s = chunk_sum();
    if (!(s < 1.15e18f)) {
        const float m_new = fmaxf(m, chunk_max());
        l *= ex2f(m - m_new);
        m = m_new;
        s = chunk_sum();
    }
    l += s;
}
template <bool kMasked, typename Release>
__device__ __forceinline__ void lse_fold(uint32_t taddr, int valid, float scale, float& m, float& l, Release release) {
#pragma unroll 1
    for (int c = 0; c < 128; c += 32) {
        float v[32];
        tmem_ld32(taddr + c, v);
        if (c == 96) release();
        if (!kMasked || valid > c) lse_chunk<kMasked>(v, valid - c, scale, m, l);
    }
}

// ---- pass B epilogue: one accumulator (this thread's token x one block of kWB window positions x n heads, a head's
// positions in consecutive columns) added to the token's total.  The logits come less the row's log-sum-exp, so the
// maximum over the heads needs no further arithmetic, and one exponential per window position follows it.
template <int kWB>
__device__ __forceinline__ float imp_fold(uint32_t taddr, int n, int wvalid, float scale) {
    float t0 = 0.f, t1 = 0.f;
#pragma unroll
    for (int c = 0; c < kWB; c += 16) {
        if (c >= wvalid) break;
        float best[16];
        tmem_ld16(taddr + c, best);
        int q = 1;
#pragma unroll 1
        for (; q + 1 < n; q += 2) {
            float x[16], y[16];
            tmem_ld16(taddr + q * kWB + c, x);
            tmem_ld16(taddr + (q + 1) * kWB + c, y);
#pragma unroll
            for (int w = 0; w < 16; ++w) best[w] = max3(best[w], x[w], y[w]);
        }
        if (q < n) {
            float x[16];
            tmem_ld16(taddr + q * kWB + c, x);
#pragma unroll
            for (int w = 0; w < 16; ++w) best[w] = fmaxf(best[w], x[w]);
        }
        const int left = wvalid - c;
#pragma unroll
        for (int w = 0; w < 16; w += 2) {
            t0 += (w < left) ? ex2f(best[w] * scale) : 0.f;
            t1 += (w + 1 < left) ? ex2f(best[w + 1] * scale) : 0.f;
        }
    }
    return t0 + t1;
}

// ---- pooled key sums on the tensor cores
// Pooling product of one staged tile: D[128 channels x 16 slots] = K_tile^T x Ind^T.  A = the tile as the TMA load
// wrote it ([token][channel], two 64-channel halves, 128-byte swizzle) read as an MN-major operand: 64 channels x 8
// tokens per swizzle atom, atoms 1024 bytes apart along the tokens and a half (16 KB) apart along the channels.
// B = the indicator matrix [slot][token], K-major like every other operand here.
constexpr uint32_t kIdescPool = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t(kIndSlots) >> 3) << 17) |
                                ((128u >> 4) << 24);
__device__ __forceinline__ void umma_pool(uint32_t tmem_d, uint32_t tile_smem, uint32_t ind_smem, bool accumulate, uint32_t leader) {
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {                     // 16 tokens per step
        const uint32_t a_addr = tile_smem + ks * 2048;
        const uint64_t da = uint64_t((a_addr >> 4) & 0x3fffu) | (uint64_t(kOpHalfBytes >> 4) << 16) |
                            (uint64_t(1024 >> 4) << 32) | (uint64_t(1) << 46) | (uint64_t(2) << 61);
        const uint64_t db = umma_desc_sw128(ind_smem + (ks >> 2) * (kIndBytes / 2) + (ks & 3) * 32);
        umma_bf16(tmem_d, da, db, kIdescPool, (accumulate || ks) ? 1u : 0u, leader);
    }
}
// Tokens 16 q .. 16 q + 15 of slot row j of an indicator matrix: ones (bf16 1.0) for the tokens [lo, hi), zeros elsewhere.
__device__ __forceinline__ void indicator_row(uint8_t* ind, int j, int q, int lo, int hi) {
    const uint32_t b0 = min(max(lo - 16 * q, 0), 16), b1 = min(max(hi - 16 * q, 0), 16);
    const uint32_t m = b1 > b0 ? (1u << b1) - (1u << b0) : 0u;
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = ((((m >> (2 * i)) & 3u) * 0x8001u) & 0x10001u) * 0x3F80u;      // two bits to the low ends of two halves
    uint8_t* row = ind + (q >> 2) * (kIndBytes / 2) + j * 128;
    *reinterpret_cast<uint4*>(row + ((((2 * q) & 7) ^ (j & 7)) << 4)) = make_uint4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<uint4*>(row + ((((2 * q + 1) & 7) ^ (j & 7)) << 4)) = make_uint4(v[4], v[5], v[6], v[7]);
}

// The sweep's table of slabs in global memory, for calls with more slabs than shared memory has room for beside the query rows.
__global__ void __launch_bounds__(1024) sweep_table_kernel(const SweepArgs a) {
    __shared__ uint32_t wsum[32];
    pdl_trigger();
    pdl_wait();
    for (int s = threadIdx.x; s < a.n_slabs; s += 1024)
        a.table[a.n_slabs + 1 + s] = a.block_table ? 0 : int(slab_row0(a.slab_off, a.cap, a.Hk, s / a.Hk, s % a.Hk));
    auto tiles = [&](int s) {
        const int room = a.block_table ? min(a.cap[s / a.Hk], a.max_pages * 128) : a.cap[s / a.Hk];
        return (min(max(a.kv_len[s], 0), room) + 127) >> 7;
    };
    cta_prefix<1024>(a.n_slabs, tiles, a.table, wsum);
}

// kTable: the table of slabs is in global memory (an instance of its own: the other one keeps its accesses to shared memory).
template <int kWB, bool kTable>
__global__ void __launch_bounds__(kSweepThreads, 1)
score_sweep_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapQ, const SweepArgs a) {
    extern __shared__ uint8_t sweep_smem_raw[];
    const uint32_t raw = smem_u32(sweep_smem_raw);
    uint8_t* qbuf = sweep_smem_raw + (((raw + 1023u) & ~1023u) - raw);           // [2 halves][R rows][128 bytes]
    const uint32_t q_half = uint32_t(a.R) * 128u;
    uint8_t* tiles = qbuf + size_t(a.R) * kRowBytes;                             // (R is a multiple of 16: 1024-byte aligned)
    uint8_t* indb = tiles + size_t(a.stages) * kOpBytes;                         // the indicator matrices of the pooling
    uint8_t* onesb = indb + (kIndBytes << a.ind_log);                                // pass B: the keys' side of the extra K step
    uint8_t* extb = onesb + 128 * kExtRow;                                       // pass B: the queries' side; pass A: [groups][blocks] (m, l)
    SweepCtl* ctl = reinterpret_cast<SweepCtl*>(extb + sweep_ext_bytes(a.R, a.RA));
    float* tokp = reinterpret_cast<float*>(ctl + 1);                             // [4 tiles][RB - 1][128] shares of a tile's tokens
    int* pref = kTable ? a.table : reinterpret_cast<int*>(tokp + 4 * (a.RB - 1) * 128);    // [n_slabs + 1] tile prefix
    int* rowb = pref + a.n_slabs + 1;                                            // [n_slabs] cache row of a slab's first token

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, cta = blockIdx.x;
    const int n_slabs = a.n_slabs, Hk = a.Hk;
    pdl_trigger();
    auto live = [&](int s) {
        const int room = a.block_table ? min(a.cap[s / Hk], a.max_pages * 128) : a.cap[s / Hk];
        return min(max(a.kv_len[s], 0), room);
    };

    if (tid == 0) {
        for (int s = 0; s < kStagesMax; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 3); }
        mbar_init(&ctl->qfull, 1);
        mbar_init(&ctl->qempty, 2);
        for (int i = 0; i < kAccAMax; ++i) mbar_init(&ctl->tfull_a[i], 1);
        for (int i = 0; i < 2 * kAccAMax; ++i) mbar_init(&ctl->tempty_a[i], 4);
        for (int i = 0; i < kAccB; ++i) mbar_init(&ctl->tfull_b[i], 1);
        for (int i = 0; i < 2 * kAccB; ++i) mbar_init(&ctl->tempty_b[i], 4);
        for (int i = 0; i < 4; ++i) mbar_init(&ctl->tokfull[i], a.RB > 1 ? 4 * (a.RB - 1) : 1);
        mbar_init(&ctl->extfull, 4);
        for (int i = 0; i < kAccB; ++i) mbar_init(&ctl->extempty[i], 2);
        for (int i = 0; i < kIndRingMax; ++i) { mbar_init(&ctl->ifull[i], kPoolWarps); mbar_init(&ctl->iempty[i], 1); }
        for (int i = 0; i < 2; ++i) mbar_init(&ctl->pfull[i], 1);
        for (int i = 0; i < 3; ++i) mbar_init(&ctl->retired[i], 1);
        ctl->abort_flag = 0;
        mbar_fence_init();
        tmap_prefetch(&mapK);
        tmap_prefetch(&mapQ);
    }
    if (warp == 1) tmem_alloc(&ctl->tmem_base, 512);
    // every key row of the extra K step is 1 in the columns that carry a query row's -lse (three bf16 pieces, half of each
    // in either 8-column piece of the row, so that a swizzle that exchanges the two makes no difference)
    if (tid < 256) *reinterpret_cast<uint4*>(onesb + tid * 16) = make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
    fence_proxy_async_smem();
    pdl_wait();                                          // the lengths may come from the kernel before this call
    const uint32_t limit = load_wait_limit(a.hdr);
    tc_fence_before();
    if (kTable) {
        __syncthreads();
    } else {
        for (int s = tid; s < n_slabs; s += kSweepThreads)
            rowb[s] = a.block_table ? 0 : int(slab_row0(a.slab_off, a.cap, Hk, s / Hk, s % Hk));
        cta_prefix<kSweepThreads>(n_slabs, [&](int s) { return (live(s) + 127) >> 7; }, pref, ctl->wsum);   // also publishes the set-up
    }
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const int T = pref[n_slabs], Ge = min(G, T);         // CTA c has the tiles [c T / Ge, (c + 1) T / Ge)
    const int t_begin = cta < Ge ? int((long long)cta * T / Ge) : T, t_end = cta < Ge ? int((long long)(cta + 1) * T / Ge) : T;
    const int ntl = t_end - t_begin;
    auto slab_of = [&](int t) {                          // last slab that starts at or before tile t
        int lo = 0, hi = n_slabs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pref[mid] <= t) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    auto owner = [&](int t) { return int(((long long)(t + 1) * Ge - 1) / T); };
    const float scale = kLog2e * rsqrtf(float(kHeadDim));
    const int n = a.Hq / Hk;
    const uint32_t ext_smem = smem_u32(extb);
    // Pass A takes the tiles of the range in the order of positions 0, 1, ..., pass B comes back from the last one.  Position p is staged at
    // p % stages in both, so pass B begins with the tiles that are still there, and every use of a stage, the first to the last, has the
    // parity of p / stages.  The pass that has the pooling products goes up.
    const bool pool_a = a.pool_a != 0;
    auto tile_at = [&](int p) { return pool_a ? t_begin + p : t_end - 1 - p; };
    const int kept = max(ntl - a.stages, 0);             // positions from here on are not loaded again
    const int rem = a.R - (a.RA - 1) * 128;              // rows of the last block
    const bool can_shift = sweep_can_shift(a.R, a.RA);
    const int slots = a.RA + (can_shift ? 1 : 0);        // sums a thread keeps in pass A: one by block, the last block's on shifted tiles apart
    const int accs = pool_a ? 3 : 4;                     // accumulators and epilogue warpgroups of pass A
    constexpr int kBarA = 1;                             // named barrier: every accumulator of pass A has been read
    const int bar_a_threads = (accs * 4 + (pool_a ? 2 : 3)) * 32;

    if (ntl > 0) {
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer: key tiles
        if (lane == 0) {
            // what depends on the slab only is kept in registers: between "stage free" and the next copy's issue nothing
            // waits on shared or global memory
            int stage = 0, slab = slab_of(tile_at(0)), lo = 0, hi = 0, row0 = 0;       // tiles [lo, hi) belong to the slab
            uint32_t lap = 0, odd = 0, used = 0;                    // position / stages; by stage: an odd number of loads, any load
            bool ok = true;
            int p = 0, step = 1;
            while (p >= 0 && ok) {
                const int t = tile_at(p);
                if (t >= hi || t < lo) {
                    while (pref[slab + 1] <= t) ++slab;
                    while (pref[slab] > t) --slab;
                    lo = pref[slab]; hi = pref[slab + 1];
                    row0 = rowb[slab];
                }
                const int j = t - lo;
                const int row = a.block_table ? max(a.block_table[size_t(slab) * a.max_pages + j], 0) * 128 : row0 + j * 128;
                const uint32_t bit = 1u << stage;
                if (used & bit) ok = role_wait(&ctl->empty[stage], (lap & 1u) ^ 1u, limit, &ctl->abort_flag, a.status);
                if (!ok) break;
                uint8_t* dst = tiles + size_t(stage) * kOpBytes;
                mbar_expect_tx(&ctl->full[stage], kOpBytes);
                tma_load_2d(dst, &mapK, 0, row, &ctl->full[stage]);
                tma_load_2d(dst + kOpHalfBytes, &mapK, 64, row, &ctl->full[stage]);
                used |= bit;
                odd ^= bit;
                if (step > 0) {
                    if (++stage == a.stages) { stage = 0; ++lap; }
                    if (++p < ntl) continue;
                    // (stage and lap stand at position ntl; position kept has the same stage a lap earlier, if any lap)
                    step = -1;
                    p = kept;
                    if (ntl >= a.stages) --lap;
                }
                if (--stage < 0) { stage = a.stages - 1; --lap; }
                --p;
            }
            // Whoever gave up: this warp stays until its copies have landed and the issuers' products have completed, so that the CTA gives
            // back shared and tensor memory with nothing in flight.
            for (int s = 0; s < a.stages; ++s)
                if ((used >> s) & 1u) mbar_wait(&ctl->full[s], ((odd >> s) & 1u) ^ 1u, kRetirePolls);
            for (int s = 0; s < 3; ++s) mbar_wait(&ctl->retired[s], 0u, kRetirePolls);
        }
    } else if (warp < 3) {
        // ------------------------------------------------------------------ MMA warps
        // Two of them take the products in turn, so that one looks at its barriers while the other's product runs.
        const uint32_t mine = warp - 1, leader = elect_leader();
        const uint32_t q0 = smem_u32(qbuf), tiles0 = smem_u32(tiles);
        bool ok = true;
        uint32_t qlap = 0, lap = 0;
        int stage = 0;
        // Both warps arrive on the stage of every tile, also where one has no product of it: a stage that was filled again before that one had
        // seen it full would leave it waiting for a phase that is two back.  The third arrival is the pooling issuer's or, in the other pass, one more here.
        auto free_stage = [&](bool has_product, bool pooled) {
            if (has_product) umma_commit(&ctl->empty[stage], leader);
            if (leader) {
                if (!has_product) mbar_arrive(&ctl->empty[stage]);
                if (!pooled && mine == 0) mbar_arrive(&ctl->empty[stage]);
            }
            __syncwarp();
        };
        {
            int slab = slab_of(tile_at(0)), lo = 0, hi = 0;
            // the next product: whose it is, its accumulator and its place in the ring of tempty
            uint32_t turn = 0, buf = 0, ring = 0, par = 1;           // par: the parity to wait for, at the place half a ring on
            bool first = true;                                       // nothing to wait for yet
            const uint32_t n_acc = accs;
            for (int p = 0; p < ntl && ok; ++p) {
                const int t = tile_at(p);
                if (t >= hi || t < lo) {
                    while (pref[slab + 1] <= t) ++slab;
                    while (pref[slab] > t) --slab;
                    lo = pref[slab]; hi = pref[slab + 1];
                    ok = warp_wait(&ctl->qfull, qlap & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    ++qlap;
                }
                // (both warps follow every tile's arrival, so that they see each phase of a stage's barrier)
                ok = warp_wait(&ctl->full[stage], lap & 1u, limit, &ctl->abort_flag, a.status);
                for (int k = 0; k < a.RA && ok; ++k) {
                    if (turn == mine) {
                        // the product n_acc before this one has been read
                        const bool upper = ring >= n_acc;
                        if (!first || upper) ok = warp_wait(&ctl->tempty_a[upper ? ring - n_acc : ring + n_acc], upper ? par ^ 1u : par, limit, &ctl->abort_flag, a.status);
                        if (!ok) break;
                        tc_fence_after();
                        const int r = k + 1 == a.RA && can_shift && (p & 1) ? a.R - 128 : k * 128;     // first query row
                        umma_tile(tmem_base + buf * 128, q0 + uint32_t(r) * 128u, q_half, tiles0 + uint32_t(stage) * kOpBytes,
                                  kOpHalfBytes, kIdescBf16M128N128, leader);
                        umma_commit(&ctl->tfull_a[buf], leader);
                    }
                    turn ^= 1u;
                    if (++buf == n_acc) buf = 0;
                    if (++ring == 2 * n_acc) { ring = 0; par ^= 1u; first = false; }
                }
                if (p + 1 < ntl) {                                   // (the last slab's rows stay for pass B)
                    const int t_next = tile_at(p + 1);
                    if (t_next >= hi || t_next < lo) umma_commit(&ctl->qempty, leader);
                }
                if (p < kept) free_stage(a.RA > 1 || turn != mine, pool_a);
                if (++stage == a.stages) { stage = 0; ++lap; }
            }
        }
        tc_fence_before();
        named_bar_sync(kBarA, bar_a_threads);
        tc_fence_after();
        if (ok) {
            int slab = slab_of(tile_at(ntl - 1)), lo = 0, hi = 0;
            uint32_t elap = 0, turn = 0, buf = 0, ring = 0, par = 1;
            bool first = true;
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t(a.N) >> 3) << 17) | ((128u >> 4) << 24);
            const uint64_t d_ones = umma_desc_sw32(smem_u32(onesb));
            for (int p = ntl - 1; p >= 0 && ok; --p) {
                const int t = tile_at(p);
                if (--stage < 0) { stage = a.stages - 1; --lap; }
                if (t >= hi || t < lo) {
                    while (pref[slab + 1] <= t) ++slab;
                    while (pref[slab] > t) --slab;
                    lo = pref[slab]; hi = pref[slab + 1];
                    if (elap > 0) {                                  // (the first slab's query rows are there)
                        ok = warp_wait(&ctl->qfull, qlap & 1u, limit, &ctl->abort_flag, a.status);
                        ++qlap;
                    }
                    if (ok) ok = warp_wait(&ctl->extfull, elap & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    ++elap;
                }
                ok = warp_wait(&ctl->full[stage], lap & 1u, limit, &ctl->abort_flag, a.status);
                for (int k = 0; k < a.RB && ok; ++k) {
                    if (turn == mine) {
                        const bool upper = ring >= kAccB;
                        if (!first || upper) ok = warp_wait(&ctl->tempty_b[upper ? ring - kAccB : ring + kAccB], upper ? par ^ 1u : par, limit, &ctl->abort_flag, a.status);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t d = tmem_base + buf * kAccCols;
                        umma_tile(d, tiles0 + uint32_t(stage) * kOpBytes, kOpHalfBytes, q0 + uint32_t(k * a.N) * 128u, q_half, idesc, leader);
                        umma_bf16(d, d_ones, umma_desc_sw32(ext_smem + uint32_t(k * a.N) * kExtRow), idesc, 1u, leader);      // - lse
                        umma_commit(&ctl->tfull_b[buf], leader);
                    }
                    turn ^= 1u;
                    if (++buf == kAccB) buf = 0;
                    if (++ring == 2 * kAccB) { ring = 0; par ^= 1u; first = false; }
                }
                if (p > 0) {
                    const int t_next = tile_at(p - 1);
                    if (t_next >= hi || t_next < lo) {                    // (the next product's group prepares the next slab)
                        umma_commit(&ctl->qempty, leader);
                        umma_commit(&ctl->extempty[buf], leader);
                    }
                }
                free_stage(a.RB > 1 || turn != mine, !pool_a);
            }
        }
        umma_commit(&ctl->retired[mine], leader);
    } else if (warp == 3) {
        // ------------------------------------------------------------------ issuer of the pooling products, TMA producer of the query rows
        // (not the tiles' producer: the rows of a slab wait until the slab before is done, which must not hold up the tiles)
        const uint32_t leader = elect_leader();
        const uint32_t indb_u32 = smem_u32(indb), tiles0 = smem_u32(tiles);
        uint32_t laps = 0;
        bool ok = true;
        int pc = 0, run = -1, slab = slab_of(tile_at(0));
        for (int pass = 0; pass < 2; ++pass) {           // (whoever gave up: everyone comes to the barrier)
            const bool pooling = (pass == 0) == pool_a;
            if (pass == 1 && !pool_a) {                  // (the pooled sums lie where the last accumulator of pass A was)
                tc_fence_before();
                named_bar_sync(kBarA, bar_a_threads);
                tc_fence_after();
            }
            int p = pass == 0 ? 0 : ntl - 1, stage = p % a.stages;
            uint32_t lap = uint32_t(p / a.stages);
            while (p >= 0 && p < ntl && ok) {
                // the part of a slab that begins at position p
                const int t = tile_at(p);
                while (pref[slab + 1] <= t) ++slab;
                while (pref[slab] > t) --slab;
                const int n_tiles = min(pref[slab + 1], t_end) - max(pref[slab], t_begin);
                if (pass == 0 || p < ntl - 1) {          // (pass B begins with the slab that is there)
                    if (laps > 0) ok = warp_wait(&ctl->qempty, (laps - 1) & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    if (leader) {
                        const int b = slab / Hk, h = slab % Hk;
                        mbar_expect_tx(&ctl->qfull, uint32_t(a.R) * kRowBytes);
                        for (int k = 0; k < a.RB; ++k)
                            for (int half = 0; half < 2; ++half)
                                tma_load_3d(qbuf + size_t(half) * q_half + size_t(k) * a.N * 128, &mapQ, half * 64, k * kWB, b * a.Hq + h * n, &ctl->qfull);
                    }
                    __syncwarp();
                    ++laps;
                }
                p += pass == 0 ? n_tiles : -n_tiles;
                for (int j = 0; j < n_tiles && pooling; ++j) {
                    ok = warp_wait(&ctl->full[stage], lap & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    int flags = 0;
                    do {
                        const int is = pc & ((1 << a.ind_log) - 1);
                        ok = warp_wait(&ctl->ifull[is], uint32_t(pc >> a.ind_log) & 1u, limit, &ctl->abort_flag, a.status);
                        if (!ok) break;
                        flags = *reinterpret_cast<volatile int*>(&ctl->ind_flags[is]);       // 1: more, 2: joins the run, 4: closes one
                        tc_fence_after();
                        if (flags & 4) umma_commit(&ctl->pfull[run & 1], leader);            // everything of the run before is issued
                        if (!(flags & 2)) ++run;
                        umma_pool(tmem_base + kPoolCol + uint32_t(run & 1) * kIndSlots, tiles0 + uint32_t(stage) * kOpBytes,
                                  indb_u32 + uint32_t(is) * kIndBytes, (flags & 2) != 0, leader);
                        umma_commit(&ctl->iempty[is], leader);
                        ++pc;
                    } while (flags & 1);
                    if (!ok) break;
                    if (pass == 1) {
                        umma_commit(&ctl->empty[stage], leader);
                        if (--stage < 0) { stage = a.stages - 1; --lap; }
                    } else {
                        if (int(lap) * a.stages + stage < kept) umma_commit(&ctl->empty[stage], leader);
                        if (++stage == a.stages) { stage = 0; ++lap; }
                    }
                }
            }
            if (pooling && ok && run >= 0) umma_commit(&ctl->pfull[run & 1], leader);
        }
        umma_commit(&ctl->retired[2], leader);
        if (laps) mbar_wait(&ctl->qfull, (laps - 1) & 1u, kRetirePolls);             // nothing in flight at the end, whoever gave up
    } else {
        // ------------------------------------------------------------------ epilogue warpgroups
        const int quarter = warp & 3;                        // tensor-memory lanes this warp may read
        const int g = (warp - 4) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t lane_addr = tmem_base + (uint32_t(quarter * 32) << 16);
        bool ok = true;
        if (g < accs) {
            // -------------------------------------------------------------- pass A: log-sum-exp, a thread per query row
            float2* part = reinterpret_cast<float2*>(extb);  // [group][slots][128] reference and sum
            float2* my = part + g * slots * 128 + row;
            const uint32_t acc = lane_addr + g * 128;
            uint32_t turn = 0;                               // products of this group so far
            int ti = 0, tk = g;                              // its next product: position and block
            while (tk >= a.RA) { tk -= a.RA; ++ti; }
            int slab = slab_of(tile_at(0));
            for (int done = 0; done < ntl;) {
                // one segment: the tiles of a slab that this CTA has
                const int t_cur = tile_at(done);
                while (pref[slab + 1] <= t_cur) ++slab;
                while (pref[slab] > t_cur) --slab;
                const int lo = pref[slab], n_tiles = min(pref[slab + 1], t_end) - max(lo, t_begin), seg_end = done + n_tiles;
                const int N = live(slab);
                for (int k = 0; k < slots; ++k) my[k * 128] = make_float2(-INFINITY, 0.f);
                while (ti < seg_end) {
                    const int valid = min(128, N - (tile_at(ti) - lo) * 128);
                    const bool sh = tk + 1 == a.RA && can_shift && (ti & 1);
                    float2* ml = my + (sh ? a.RA : tk) * 128;
                    float2 x = *ml;
                    if (ok) ok = warp_wait(&ctl->tfull_a[g], turn & 1u, limit, &ctl->abort_flag, a.status);
                    if (ok) {
                        tc_fence_after();
                        auto release = [&]() {               // this warp's loads of the accumulator have completed
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&ctl->tempty_a[g + (turn & 1u) * accs]);
                        };
                        // (the last block may hold fewer rows than lanes)
                        if (tk + 1 < a.RA || (sh ? quarter * 32 + 31 >= 128 - rem : quarter * 32 < rem)) {
                            if (valid == 128) lse_fold<false>(acc, valid, scale, x.x, x.y, release);
                            else              lse_fold<true>(acc, valid, scale, x.x, x.y, release);
                            *ml = x;
                        } else {
                            release();
                        }
                    }
                    ++turn;
                    tk += accs;
                    while (tk >= a.RA) { tk -= a.RA; ++ti; }
                }
                if (seg_end == ntl) {
                    tc_fence_before();
                    named_bar_arrive(kBarA, bar_a_threads);          // (the issuers go on to pass B)
                }
                named_bar_sync(2, accs * 128);
                float2* rec = a.rec + size_t(cta + slab) * (size_t(a.RA) * 128);
                for (int k = g; k < a.RA; k += accs) {       // the groups' parts -> one record per CTA and slab
                    float M = -INFINITY, L = 0.f;
                    // (the largest reference first: a sum that is rescaled on the way is rounded on the way)
                    const int n_part = can_shift && k + 1 == a.RA ? 2 * accs : accs;       // odd ones: the last block on shifted tiles
                    auto at = [&](int q) {
                        const bool sh = n_part > accs && (q & 1);
                        const int g_ = n_part > accs ? q >> 1 : q;
                        return part[(g_ * slots + (sh ? a.RA : k)) * 128 + (sh ? min(row + 128 - rem, 127) : row)];
                    };
#pragma unroll 1
                    for (int q = 0; q < n_part; ++q) M = fmaxf(M, at(q).x);
#pragma unroll 1
                    for (int q = 0; q < n_part; ++q) {
                        const float2 x = at(q);
                        L += x.y > 0.f ? x.y * ex2f(x.x - M) : 0.f;
                    }
                    rec[k * 128 + row] = make_float2(M, L);
                }
                named_bar_sync(4, accs * 128);               // the parts have been read, the record is written
                if (tid == 128 && ok) { __threadfence(); atomicAdd(a.lse_cnt + slab, uint32_t(n_tiles)); }
                done = seg_end;
            }
        }
        if (g < 3) {
            // -------------------------------------------------------------- pass B: importance, a thread per token
            // (what depends on the slab only is kept in registers: while the tensor core streams its operands every look at
            // shared memory takes a hundred cycles and more)
            const uint32_t acc = lane_addr + g * kAccCols;
            uint32_t turn = 0;                               // products of this group so far
            int slab = slab_of(tile_at(ntl - 1)), lo = 0, hi = 0, N = 0;        // the slab's tiles are [lo, hi)
            uint32_t ext_no = 0;                             // slabs begun so far
            uint32_t ext_par = 0;                            // parity of this group's next phase of extempty
            float *imp_ws = nullptr, *imp_user = nullptr;
            float out_scale = 0.f;                           // 2^-e / window of the slab
            int i = 0, k = g;                                // this group's next product: tile in the order of the pass, and block
            auto next_product = [&](int n) {
                for (k += n; k >= a.RB; k -= a.RB) ++i;
            };
            for (next_product(0); i < ntl; next_product(kAccB)) {
                const int t = tile_at(ntl - 1 - i);
                bool begins = false;
                if (t >= hi || t < lo) {
                    do {                                     // (past slabs of which this group has no product)
                        const int at = ext_no == 0 ? tile_at(ntl - 1) : pool_a ? lo - 1 : hi;
                        while (pref[slab + 1] <= at) ++slab;
                        while (pref[slab] > at) --slab;
                        lo = pref[slab]; hi = pref[slab + 1];
                        ++ext_no;
                    } while (t >= hi || t < lo);
                    N = live(slab);
                    out_scale = __uint_as_float(uint32_t(127 - lse_shift(N)) << 23) / float(a.window);
                    imp_ws = a.tok_imp_ws + size_t(slab) * a.max_cap;
                    imp_user = a.tok_imp_user ? a.tok_imp_user + (a.block_table ? size_t(slab) * a.max_pages * 128 : size_t(rowb[slab])) : nullptr;
                    begins = k == 0 && t == (pool_a ? min(hi, t_end) - 1 : max(lo, t_begin));
                }
                if (begins) {
                    // the group of a slab's first product prepares the slab: log-sum-exp of its query rows from the records of
                    // all its CTAs, negated, in units of raw logits, as three bf16 pieces of the extra K step
                    const int fc = owner(lo), lc = owner(hi - 1);
                    if (ok) ok = warp_flag_wait(a.lse_cnt + slab, uint32_t(hi - lo), limit, &ctl->abort_flag, a.status);
                    if (ok && ext_no > 1) {
                        ok = role_wait(&ctl->extempty[g], ext_par, limit, &ctl->abort_flag, a.status);
                        ext_par ^= 1u;
                    }
                    ok = __all_sync(0xffffffffu, ok);
                    if (ok) {
                        const float2* r0 = a.rec + size_t(fc + slab) * (size_t(a.RA) * 128);
                        const int n_part = lc - fc + 1;
                        for (int r = row; r < a.R; r += 128) {
                            float M = -INFINITY, L = 0.f;
                            for (int p0 = 0; p0 < n_part; p0 += 4) {         // four records per round: their loads are in flight together
                                float2 x[4];
#pragma unroll
                                for (int p = 0; p < 4; ++p)
                                    x[p] = p0 + p < n_part ? __ldcg(r0 + size_t(p0 + p) * (a.RA * 128) + r) : make_float2(-INFINITY, 0.f);
                                float mx = M;
#pragma unroll
                                for (int p = 0; p < 4; ++p) mx = fmaxf(mx, x[p].x);
                                L *= M == -INFINITY ? 0.f : ex2f(M - mx);
                                M = mx;
#pragma unroll
                                for (int p = 0; p < 4; ++p) L += x[p].y > 0.f ? x[p].y * ex2f(x[p].x - M) : 0.f;
                            }
                            // (the exponent of the sum apart, so that neither its logarithm nor the total is rounded at a larger magnitude)
                            const int ex = int(__float_as_uint(L) >> 23) - 127;
                            const float mant = __uint_as_float((__float_as_uint(L) & 0x007fffffu) | 0x3f800000u);
                            const float v = L > 0.f ? -0.5f * ((M + float(ex - lse_shift(N))) + log2f(mant)) / scale : 0.f;
                            const __nv_bfloat16 b0 = __float2bfloat16_rn(v);
                            const float v1 = v - __bfloat162float(b0);
                            const __nv_bfloat16 b1 = __float2bfloat16_rn(v1), b2 = __float2bfloat16_rn(v1 - __bfloat162float(b1));
                            const uint4 piece = make_uint4(uint32_t(__bfloat16_as_ushort(b0)) | (uint32_t(__bfloat16_as_ushort(b1)) << 16),
                                                           uint32_t(__bfloat16_as_ushort(b2)), 0u, 0u);
                            *reinterpret_cast<uint4*>(extb + size_t(r) * kExtRow) = piece;
                            *reinterpret_cast<uint4*>(extb + size_t(r) * kExtRow + 16) = piece;
                        }
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&ctl->extfull);
                    }
                }
                if (ok) ok = warp_wait(&ctl->tfull_b[g], turn & 1u, limit, &ctl->abort_flag, a.status);
                if (!ok) continue;
                tc_fence_after();
                float total = imp_fold<kWB>(acc, n, min(kWB, a.window - k * kWB), scale);
                float* share = tokp + (i & 3) * (a.RB - 1) * 128 + row;
                if (k + 1 < a.RB) {
                    share[k * 128] = total;                  // another group adds the shares up, in the order of the blocks
                } else if (a.RB > 1) {
                    ok = warp_wait(&ctl->tokfull[i & 3], uint32_t(i >> 2) & 1u, limit, &ctl->abort_flag, a.status);
                    for (int q = a.RB - 2; q >= 0; --q) total += share[q * 128];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (k + 1 < a.RB) mbar_arrive(&ctl->tokfull[i & 3]);
                    mbar_arrive(&ctl->tempty_b[g + (turn & 1u) * kAccB]);
                }
                ++turn;
                const int tok = (t - lo) * 128 + row;
                if (k + 1 == a.RB && ok && tok < N) {
                    const float v = total * out_scale;
                    imp_ws[tok] = v;
                    if (imp_user) imp_user[tok] = v;
                }
            }
        } else {
            // -------------------------------------------------------------- per-sentence sums of the key rows
            // The sums are a product on the tensor cores: (tile^T: channel x token) x (indicator: token x sentence slot).
            // A run of consecutive tiles whose sentences all fall among the 16 sentences B .. B + 15 shares one accumulator
            // (slot j = sentence B + j; the products of the run accumulate), so the sums are read out and stored to global
            // memory once per run, about every fifth tile.  Each of the four warps writes a quarter of a tile's matrix and
            // arrives; a fifth warp issues the product.  A tile that touches more than 16 sentences (empty ones count) gets several
            // matrices, each a run of its own.
            // The matrices depend on the sentence offsets alone, so they run ahead of the tiles, as far as their ring goes.  Every
            // warp keeps, one entry per lane, the offsets B .. B + 31 of the current run (entries past the table read as "never
            // starts"), from which a run's length, its sentences and the next run's first sentence follow at once; the next run's offsets
            // are fetched while this one's matrices are written.  (With the run worked out tile by tile, behind the tile's arrival, a tile took
            // these warps 2260 clocks and pass A 1.15 us.)
            // A sentence that began in an earlier run of this CTA is added to; one that began before the CTA's range belongs to the CTA in whose
            // range it began: its part is kept until every CTA of the slab has stored its sums, and added then.  So nothing has to be cleared.
            constexpr int kNever = 0x7fffffff;
            const int gw = quarter;                               // warp of the group: slots 4 gw .. 4 gw + 3 of a matrix
            const int gtid = tid - 512;
            const int ch = row;
            const int sj = 4 * gw + (lane >> 3), sq = lane & 7;     // this thread writes tokens 16 sq .. 16 sq + 15 of slot row sj
            const int ring = (1 << a.ind_log) - 1;
            int slab = slab_of(t_begin), lo = 0, hi = 0, S = 0, N = 0;      // the slab's tiles are [lo, hi)
            const int slab_first = slab;
            const int32_t* so = a.sent_off;
            int t = t_begin, ic = 0, run = 0;                       // next tile, matrices written, runs opened
            int B = 0, w = kNever;                                  // the run's first sentence, offset of sentence B + lane
            float head = 0.f;
            int head_sent = -1;
            // 32-way search for the last sentence that starts at or before token `tok`, one probe per lane
            auto holder = [&](int tok) {
                int first = 0, len = S;
                while (len > 32) {
                    const int stride = (len + 31) >> 5;
                    const int pidx = first + lane * stride;
                    const bool le = pidx < first + len && so[pidx] <= tok;
                    const int adv = max(__popc(__ballot_sync(0xffffffffu, le)) - 1, 0) * stride;
                    len = min(stride, len - adv);
                    first += adv;
                }
                const bool le = lane < len && so[first + lane] <= tok;
                return first + max(__popc(__ballot_sync(0xffffffffu, le)) - 1, 0);
            };
            auto fetch = [&](int first) { return first + lane <= S ? so[first + lane] : kNever; };
            // the run before, to be read out: its slab, first sentence, slots that hold tokens; where its first sentence began (0: in it, 1: in an
            // earlier run, 2: before the CTA's range); where it is the last of a slab, the tiles that this CTA has of it
            int p_slab = 0, p_B = 0, p_from = 0, p_tiles = 0;
            uint32_t p_held = 0;
            auto drain = [&](int r) {                               // (accumulator r & 1)
                ok = warp_wait(&ctl->pfull[r & 1], uint32_t(r >> 1) & 1u, limit, &ctl->abort_flag, a.status);
                if (!ok) return;
                tc_fence_after();
                float v[kIndSlots];
                tmem_ld16(lane_addr + kPoolCol + uint32_t(r & 1) * kIndSlots, v);
                tc_fence_before();
                float* dst = a.vsum + (size_t(p_slab) * a.max_sent + p_B) * kHeadDim + ch;
                if (p_held & 1u) {
                    if (p_from == 2) { head += v[0]; head_sent = p_B; }
                    else if (p_from == 1) atomicAdd(dst, v[0]);
                    else *dst = v[0];
                }
#pragma unroll
                for (int j = 1; j < kIndSlots; ++j)
                    if (p_held & (1u << j)) dst[size_t(j) * kHeadDim] = v[j];
                if (p_tiles > 0) {
                    __syncwarp();
                    if (lane == 0) { __threadfence(); atomicAdd(a.sum_cnt + p_slab, uint32_t(p_tiles)); }
                }
            };
            while (t < t_end && ok) {
                if (t >= hi) {
                    while (pref[slab + 1] <= t) ++slab;
                    lo = pref[slab]; hi = pref[slab + 1];
                    so = a.sent_off + size_t(slab) * (a.max_sent + 1);
                    S = min(max(a.n_sent[slab], 0), a.max_sent);
                    N = live(slab);
                    B = t > lo ? holder((t - lo) * 128) : 0;        // (a slab that opens with empty sentences: they get slots)
                    w = fetch(B);
                }
                // the run: all tiles that end at or before sentence B + 16 begins, at least one
                const int tok0 = (t - lo) * 128, last_tile = min(hi, t_end);
                const int stop = B + kIndSlots < S ? __shfl_sync(0xffffffffu, w, kIndSlots) : kNever;
                const int fit = stop >= N ? last_tile - t : min(last_tile - t, max(stop - tok0, 0) >> 7);
                const int more = fit == 0 ? 1 : 0, n_tiles = max(fit, 1);           // more: slot 15 leaves some of the tile
                const int tok_end = min(tok0 + n_tiles * 128, N);
                const int w1 = __shfl_down_sync(0xffffffffu, w, 1);
                const uint32_t held = __ballot_sync(0xffffffffu, lane < kIndSlots && B + lane < S && min(w1, tok_end) > max(w, tok0));
                const int began = __shfl_sync(0xffffffffu, w, 0);
                int wj = __shfl_sync(0xffffffffu, w, sj), wj1 = __shfl_sync(0xffffffffu, w, sj + 1);    // this thread's slot row
                if (B + sj >= S) wj = wj1 = kNever;
                // the next run: in the same tile, or in the last sentence that starts at or before the next tile's first token
                int B_next = B + kIndSlots, w_next = kNever;
                if (!more && t + n_tiles < last_tile) {
                    const int n_le = __popc(__ballot_sync(0xffffffffu, B + lane < S && w <= tok_end));
                    B_next = (n_le == 32 && B + 32 < S) ? holder(tok_end) : B + max(n_le - 1, 0);
                }
                if (more || t + n_tiles < last_tile) w_next = fetch(B_next);
                for (int k = 0; k < n_tiles && ok; ++k, ++ic) {
                    const int tok = tok0 + k * 128, valid = min(128, N - tok), is = ic & ring;
                    if (valid < 128) {
                        // This matrix needs its tile: a zero in the indicator does not silence a NaN or an infinity in a dead row, so the rows
                        // past the slab's end are cleared in the staged tile (the logits of those rows are never read).  Once the last
                        // matrix has been multiplied, all tiles before this one had arrived, so the wait is for the right phase of the stage.
                        if (ic > 0) ok = warp_wait(&ctl->iempty[(ic - 1) & ring], uint32_t((ic - 1) >> a.ind_log) & 1u, limit, &ctl->abort_flag, a.status);
                        const int i = pool_a ? t + k - t_begin : t_end - 1 - (t + k), stage = i % a.stages;
                        if (ok) ok = warp_wait(&ctl->full[stage], uint32_t(i / a.stages) & 1u, limit, &ctl->abort_flag, a.status);
                        if (!ok) break;
                        uint8_t* tile = tiles + size_t(stage) * kOpBytes;
                        for (int u = valid * 8 + gtid; u < 128 * 8; u += kPoolWarps * 32) {
                            *reinterpret_cast<uint4*>(tile + u * 16) = make_uint4(0u, 0u, 0u, 0u);
                            *reinterpret_cast<uint4*>(tile + kOpHalfBytes + u * 16) = make_uint4(0u, 0u, 0u, 0u);
                        }
                    } else if (ic >> a.ind_log) {                   // the product that read this buffer last has completed
                        ok = warp_wait(&ctl->iempty[is], uint32_t((ic >> a.ind_log) - 1) & 1u, limit, &ctl->abort_flag, a.status);
                        if (!ok) break;
                    }
                    indicator_row(indb + size_t(is) * kIndBytes, sj, sq, min(max(wj - tok, 0), valid), min(max(wj1 - tok, 0), valid));
                    fence_proxy_async_smem();                       // the matrix (and cleared rows) are read by the tensor core
                    tc_fence_before();                              // and this warp's reads of the accumulators came first
                    __syncwarp();
                    if (lane == 0) {
                        if (gw == 0) ctl->ind_flags[is] = more | (k > 0 ? 2 : 0) | (k == 0 && run > 0 ? 4 : 0);
                        mbar_arrive(&ctl->ifull[is]);
                    }
                    if (k == (n_tiles > 1 ? 1 : 0) && run > 0) drain(run - 1);      // the run before, while this one is multiplied
                }
                p_slab = slab; p_B = B; p_held = held;
                p_from = began < max(t_begin - lo, 0) * 128 ? 2 : began < tok0 ? 1 : 0;
                p_tiles = !more && t + n_tiles == last_tile ? last_tile - max(lo, t_begin) : 0;
                ++run;
                if (!more) t += n_tiles;
                B = B_next; w = w_next;
            }
            if (ok && run > 0) drain(run - 1);                      // (the issuer closes the last run when its tiles are done)
            if (ok && head_sent >= 0) {
                const uint32_t all = 4u * uint32_t(pref[slab_first + 1] - pref[slab_first]);
                if (warp_flag_wait(a.sum_cnt + slab_first, all, limit, &ctl->abort_flag, a.status))
                    atomicAdd(a.vsum + (size_t(slab_first) * a.max_sent + head_sent) * kHeadDim + ch, head);
            }
        }
    }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ---------------------------------------------------------------------------------------
// pooling: a warp takes kPoolRows sentences, 4 channels per lane; writes the normalised mean key as bf16 hi + lo.
// Bound by DRAM where there are many sentences (512 bytes in and out each): the loads of all the warp's sentences are in flight
// together, importances of the first 96 tokens included.
// ---------------------------------------------------------------------------------------
constexpr int kPoolRows = 4;
__global__ void __launch_bounds__(256)
score_pool_kernel(uint32_t* lse_cnt, int Hk, int max_sent, int max_cap, int max_rows, const int32_t* cap, const int32_t* kv_len,
                  const int32_t* sent_off, const int32_t* n_sent, float eps, const float* tok_imp_ws,
                  const float* vsum, float* sent_imp, __nv_bfloat16* vbar_hi, __nv_bfloat16* vbar_lo, float* sent_lam) {
    pdl_trigger();
    pdl_wait();
    const int slab = blockIdx.y;
    if (blockIdx.x == 0 && threadIdx.x < 2) lse_cnt[threadIdx.x * gridDim.y + slab] = 0u;      // both counters, for the next call's sweeps
    const int lane = threadIdx.x & 31;
    const int i0 = blockIdx.x * 8 * kPoolRows + (threadIdx.x >> 5);         // and every eighth after it
    const int S = min(max(n_sent[slab], 0), max_sent);
    const int N = min(max(kv_len[slab], 0), min(cap[slab / Hk], max_rows));
    const int32_t* so = sent_off + size_t(slab) * (max_sent + 1);
    const float* imp = tok_imp_ws + size_t(slab) * max_cap;
    int b[kPoolRows], e[kPoolRows];
    float4 v[kPoolRows];
#pragma unroll
    for (int q = 0; q < kPoolRows; ++q) {
        const int i = i0 + q * 8;
        b[q] = e[q] = 0;
        v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < S) {
            b[q] = max(so[i], 0);
            e[q] = min(so[i + 1], N);
            v[q] = reinterpret_cast<const float4*>(vsum + (size_t(slab) * max_sent + i) * kHeadDim)[lane];
        }
    }
    float first[kPoolRows][3];
#pragma unroll
    for (int q = 0; q < kPoolRows; ++q)
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const int t = b[q] + p * 32 + lane;
            first[q][p] = t < e[q] ? imp[t] : 0.f;
        }
#pragma unroll
    for (int q = 0; q < kPoolRows; ++q) {
        const int i = i0 + q * 8;
        if (i >= S) {                                        // the rest of the last block: zeros, whose products are finite
            if (i < min((S + 127) / 128 * 128, max_sent)) {
                const size_t o = (size_t(slab) * max_sent + i) * kHeadDim;
                reinterpret_cast<uint2*>(vbar_hi + o)[lane] = reinterpret_cast<uint2*>(vbar_lo + o)[lane] = make_uint2(0u, 0u);
            }
            continue;
        }
        float ti = first[q][0] + first[q][1] + first[q][2];
        for (int t = b[q] + 96 + lane; t < e[q]; t += 32) ti += imp[t];
        const float len = float(max(e[q] - b[q], 1));
        if (e[q] <= b[q]) v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        const float m[4] = {v[q].x / len, v[q].y / len, v[q].z / len, v[q].w / len};
        float nn = m[0] * m[0] + m[1] * m[1] + m[2] * m[2] + m[3] * m[3];
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            nn += __shfl_xor_sync(0xffffffffu, nn, d);
            ti += __shfl_xor_sync(0xffffffffu, ti, d);
        }
        const float inv = 1.f / (sqrtf(nn) + eps);
        uint32_t hi[4], lo[4];                               // bf16 bit patterns
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float x = m[c] * inv;
            const __nv_bfloat16 h = __float2bfloat16_rn(x);
            const __nv_bfloat16 r = __float2bfloat16_rn(x - __bfloat162float(h));
            hi[c] = __bfloat16_as_ushort(h);
            lo[c] = __bfloat16_as_ushort(r);
        }
        const size_t o = (size_t(slab) * max_sent + i) * kHeadDim;
        reinterpret_cast<uint2*>(vbar_hi + o)[lane] = make_uint2(hi[0] | (hi[1] << 16), hi[2] | (hi[3] << 16));
        reinterpret_cast<uint2*>(vbar_lo + o)[lane] = make_uint2(lo[0] | (lo[1] << 16), lo[2] | (lo[3] << 16));
        if (lane == 0) {
            const size_t s = size_t(slab) * max_sent + i;
            sent_imp[s] = (e[q] > b[q]) ? ti / len : 0.f;
            sent_lam[s] = 0.f;                               // (as bits: below every ordered penalty)
        }
    }
}

// ---------------------------------------------------------------------------------------
// Gram passes on the tensor cores.  G is symmetric: every pair of 128-sentence blocks I <= J of a slab is multiplied and
// exponentiated once, and gives the rows of I their sums over the columns and the columns of J theirs over the rows (the
// diagonal pair: column sums only).  Work is the list of pairs, J by J, over all slabs, cut into equal contiguous ranges.
// A column block's sums are kept for as long as a range stays with it and stored as that part's (four warps' each); a row's are stored by pair (four column
// groups).  The CTA that completes a slab adds a sentence's parts and rows up in order, so the results do not depend on who was first.
// They lie where the sums of the keys were, which the pooling was the last to read.
// Rows past a slab's last sentence are zeros (written, or beyond the table and filled in by the copy), so nothing is masked but the weights of such
// columns and, in a diagonal pair, a sentence's product with itself.
// The penalty is the maximum over later sentences; only those beyond tau are reported, which are few (pass 1, an integer maximum).
// Roles as in the token-level kernel: a TMA warp, two MMA warps that take the pairs in turn, sixteen epilogue warps with 32
// rows x 32 columns of every accumulator each, column sums in registers for as long as J stays.
// Three shared-memory slots hold a block's high and low parts.  One is J's, the other two take the I blocks in turn; the next J takes
// the slot that is free next and the old J's goes to the end of the queue, so a change of J costs no drain.
// What counts is the epilogue's instructions, 32 exponentials and about 60 others per warp and pair: with the walk over the pairs, addresses, zeros
// for parts that a pair did not have, masks and reciprocals in the loop it was 1790 and 1380 a scheduler and pair (passes 1 and 2), now
// 1310 and 1140, and 306 and 271 us became 230 and 227 (kernel times, 128 slabs x 2K sentences).  Of the 1.75 us a pair the three products,
// which stream 192 KB of operands at the shared-memory port's 128 bytes per clock, take 0.8; the 64 KB of a pair's I block are
// 5.5 TB/s from L2 over all SMs.
// ---------------------------------------------------------------------------------------
constexpr int kGramAcc = 4;
struct GramCtl {
    uint64_t full[3][2], empty[3][2];        // slot, part: loaded (every use) / given back by the pair that used it as I
    uint64_t ddone[3];                       // the diagonal pair of the J block in this slot is complete
    uint64_t turn[2];
    uint64_t tfull[kGramAcc], tempty[kGramAcc];
    uint32_t tmem_base;
    int abort_flag, last;
    uint32_t wsum[32];
    alignas(16) float colw[16][32];          // by epilogue warp: weights of its columns, 1 or (pass 2) 1 / Z_j, 0 for none of the slab's
    uint64_t retired[2];                     // every product of an MMA warp has completed
    uint32_t loads[6];                       // by slot and part: copies issued (in shared memory for want of registers)
};
constexpr int kGramThreads = 20 * 32;        // TMA warp, two MMA warps, one idle, four epilogue warpgroups
static size_t gram_smem_bytes(int slabs) { return 1024 + 6 * size_t(kOpBytes) + sizeof(GramCtl) + size_t(slabs + 1) * 4; }

// Floats as integers in the same order (0 lies below all of them).
__device__ __forceinline__ uint32_t ordered_bits(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_ordered_bits(uint32_t u) { return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u); }

// A CTA's walk over its pairs, and which slot a block is in.  Every role steps through the same sequence.
struct GramWalk {
    int slab, J, t;                          // pair t of block column J: 0 is the diagonal, t > 0 multiplies block t - 1
    int left;                                // pairs of the range not yet walked, this one included
    int jslot, q0, q1, q2;                   // slot of J, and the others in the order in which they are taken
    bool have_j;
    __device__ __forceinline__ void start(const int* ipref, int first, int count) {
        left = count; slab = 0; have_j = false; q0 = 0; q1 = 1; q2 = 2; jslot = 0;
        if (count <= 0) return;
        while (ipref[slab + 1] <= first) ++slab;
        const int p = first - ipref[slab];
        J = int((sqrtf(8.f * float(p) + 1.f) - 1.f) * 0.5f);
        while (J > 0 && J * (J + 1) / 2 > p) --J;
        while ((J + 1) * (J + 2) / 2 <= p) ++J;
        t = p - J * (J + 1) / 2;
    }
    __device__ __forceinline__ int pop() { const int s = q0; q0 = q1; q1 = q2; return s; }
    __device__ __forceinline__ void take_j() {           // J changes (or the range begins)
        if (have_j) q2 = jslot;                          // the old one's slot goes to the end of the queue
        jslot = pop();
        have_j = true;
    }
    __device__ __forceinline__ int take_i() { const int s = pop(); q1 = s; return s; }
    // on to the next pair: true if it has another J
    __device__ __forceinline__ bool next(const int* ipref) { return advance(ipref, 1); }
    // on by n pairs, at most to the next J
    __device__ __forceinline__ bool advance(const int* ipref, int n) {
        left -= n;
        t += n;
        if (t <= J) return false;
        t = 0; ++J;
        if (left > 0 && ipref[slab] + J * (J + 1) / 2 >= ipref[slab + 1]) {
            J = 0;
            do ++slab; while (ipref[slab + 1] == ipref[slab]);
        }
        return true;
    }
};

// Optional source of the sentence penalty: the lookup table T of one value per generation-space sentence,
// [batch][table_len], read through the cache-space sentence's generation-space index (Phi).  table == nullptr:
// the penalty comes from the pooled keys of the slab.
struct LamTable {
    const float* table;
    const int32_t* sent_id;
    int table_len;
    int Hk;
};

template <int kPass>
__global__ void __launch_bounds__(kGramThreads, 1)
score_gram_kernel(const __grid_constant__ CUtensorMap mapHi, const __grid_constant__ CUtensorMap mapLo, int n_slabs,
                  int max_sent, const int32_t* n_sent, float sigma, float tau, float* sc_z, const float* sent_imp,
                  float* sent_red, float* sent_lam, float* sent_score, float* parts, size_t parts_slab, uint32_t* cnt, LamTable ext, const Header* hdr) {
    extern __shared__ uint8_t gram_smem_raw[];
    const uint32_t raw = smem_u32(gram_smem_raw);
    uint8_t* slots = gram_smem_raw + (((raw + 1023u) & ~1023u) - raw);           // 3 x (high, low)
    GramCtl* ctl = reinterpret_cast<GramCtl*>(slots + 6 * kOpBytes);
    int* ipref = reinterpret_cast<int*>(ctl + 1);                                // [n_slabs + 1] prefix of pairs
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto sent_of = [&](int s) { return min(max(n_sent[s], 0), max_sent); };
    pdl_trigger();

    if (tid == 0) {
        for (int s = 0; s < 3; ++s) {
            for (int part = 0; part < 2; ++part) { mbar_init(&ctl->full[s][part], 1); mbar_init(&ctl->empty[s][part], 1); }
            mbar_init(&ctl->ddone[s], 1);
        }
        for (int s = 0; s < 2; ++s) { mbar_init(&ctl->turn[s], 1); mbar_init(&ctl->retired[s], 1); }
        for (int s = 0; s < kGramAcc; ++s) { mbar_init(&ctl->tfull[s], 1); mbar_init(&ctl->tempty[s], 16); }
        ctl->abort_flag = 0;
        mbar_fence_init();
        tmap_prefetch(&mapHi);
        tmap_prefetch(&mapLo);
    }
    if (warp == 1) tmem_alloc(&ctl->tmem_base, 128 * kGramAcc);
    pdl_wait();                                          // n_sent, the pooled keys and the row sums may come from the kernel before
    uint32_t* status = const_cast<uint32_t*>(&hdr->status);
    const uint32_t limit = load_wait_limit(hdr);
    tc_fence_before();
    cta_prefix<kGramThreads>(n_slabs, [&](int s) { const int nb = (sent_of(s) + 127) >> 7; return nb * (nb + 1) / 2; }, ipref, ctl->wsum);
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const long long total = ipref[n_slabs];
    const int ctas = int(min((long long)gridDim.x, total)), cta = min(int(blockIdx.x), ctas);          // none of those with work has no pair
    const int first = ctas > 0 ? int(total * cta / ctas) : 0, count = int(blockIdx.x) < ctas ? int(total * (cta + 1) / ctas) - first : 0;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        if (warp == 0 && lane == 0) {
            bool ok = true;
            uint32_t ipar = 0, lasti = 0, dpar = 0, lastd = 0;         // bits by slot
            ctl->loads[0] = ctl->loads[1] = ctl->loads[2] = ctl->loads[3] = ctl->loads[4] = ctl->loads[5] = 0;
            GramWalk w;
            w.start(ipref, first, count);
            auto load = [&](int s, int block) {
                // What used the slot last: an I block gives its parts back one by one.  A J block was in use until its last pair, and the
                // pairs with an I have given their slots back by now (both others were taken since); the diagonal one is waited for here.
                const bool was_i = (lasti >> s) & 1u;
                if ((lastd >> s) & 1u) ok = role_wait(&ctl->ddone[s], ((dpar >> s) & 1u) ^ 1u, limit, &ctl->abort_flag, status);
                for (int part = 1; part >= 0 && ok; --part) {             // low, high: the order in which they are given back
                    if (was_i) ok = role_wait(&ctl->empty[s][part], ((ipar >> s) & 1u) ^ 1u, limit, &ctl->abort_flag, status);
                    if (!ok) break;
                    uint8_t* dst = slots + size_t(2 * s + part) * kOpBytes;
                    const CUtensorMap* map = part ? &mapLo : &mapHi;
                    mbar_expect_tx(&ctl->full[s][part], kOpBytes);
                    tma_load_3d(dst, map, 0, block * 128, w.slab, &ctl->full[s][part]);
                    tma_load_3d(dst + kOpHalfBytes, map, 64, block * 128, w.slab, &ctl->full[s][part]);
                    ++ctl->loads[2 * s + part];
                }
            };
            bool fresh = true;
            while (w.left > 0 && ok) {
                if (fresh) {
                    w.take_j();
                    load(w.jslot, w.J);
                    const uint32_t bit = 1u << w.jslot;
                    lasti &= ~bit;
                    lastd = w.t == 0 ? lastd | bit : lastd & ~bit;
                    if (w.t == 0) dpar ^= bit;                        // parity of the next diagonal in this slot
                }
                if (w.t > 0 && ok) {
                    const int s = w.take_i();
                    load(s, w.t - 1);
                    lasti |= 1u << s;
                    lastd &= ~(1u << s);
                    ipar ^= 1u << s;
                }
                fresh = w.next(ipref);
            }
            // Whoever gave up: this warp stays until its copies have landed and the issuers' products have completed, so that the CTA gives
            // back shared and tensor memory with nothing in flight.
            for (int s = 0; s < 3; ++s)
                for (int part = 0; part < 2; ++part)
                    if (ctl->loads[2 * s + part]) mbar_wait(&ctl->full[s][part], (ctl->loads[2 * s + part] - 1) & 1u, kRetirePolls);
            for (int s = 0; s < 2; ++s) mbar_wait(&ctl->retired[s], 0u, kRetirePolls);
        } else if (warp == 1 || warp == 2) {
            // A pair each in turn, so that one waits for its operands while the other's products run.  The turn is handed over a little
            // before a pair's last instructions are issued.  It comes before the other waits: every barrier's earlier phases have been seen by then.
            const uint32_t me = warp - 1, leader = elect_leader();
            bool ok = true, fresh = true;
            uint32_t fpar = 0, jpar = 0;                               // parity of a slot's next use; of J's present one
            GramWalk w;
            w.start(ipref, first, count);
            for (uint32_t bc = 0; w.left > 0 && ok; ++bc) {
                if (fresh) {
                    w.take_j();
                    jpar = (fpar >> w.jslot) & 1u;
                    fpar ^= 1u << w.jslot;
                }
                int is = w.jslot;
                uint32_t ip = jpar;
                const bool diag = w.t == 0;
                if (!diag) {
                    is = w.take_i();
                    ip = (fpar >> is) & 1u;
                    fpar ^= 1u << is;
                }
                const int js = w.jslot;
                fresh = w.next(ipref);
                if ((bc & 1u) != me) continue;
                const uint32_t acc = bc % kGramAcc;
                if (bc > 0) ok = warp_wait(&ctl->turn[me], ((bc >> 1) - (me ? 0u : 1u)) & 1u, limit, &ctl->abort_flag, status);
                for (int part = 1; part >= 0 && ok; --part) {
                    ok = warp_wait(&ctl->full[js][part], jpar, limit, &ctl->abort_flag, status);
                    if (ok && !diag) ok = warp_wait(&ctl->full[is][part], ip, limit, &ctl->abort_flag, status);
                }
                if (ok && bc >= kGramAcc) ok = warp_wait(&ctl->tempty[acc], ((bc / kGramAcc) - 1) & 1u, limit, &ctl->abort_flag, status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t i_hi = smem_u32(slots + size_t(2 * is) * kOpBytes), j_hi = smem_u32(slots + size_t(2 * js) * kOpBytes);
                const uint32_t d = tmem_base + acc * 128;
                umma_tile_128x128x128(d, i_hi + kOpBytes, j_hi, false, leader);
                if (!diag) umma_commit(&ctl->empty[is][1], leader);
                umma_tile_128x128x128(d, i_hi, j_hi + kOpBytes, true, leader);
                if (leader) mbar_arrive(&ctl->turn[me ^ 1u]);
                __syncwarp();
                umma_tile_128x128x128(d, i_hi, j_hi, true, leader);
                umma_commit(&ctl->tfull[acc], leader);
                umma_commit(diag ? &ctl->ddone[js] : &ctl->empty[is][0], leader);
            }
            umma_commit(&ctl->retired[me], leader);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        const int quarter = warp & 3, cg = (warp - 4) >> 2, c0 = cg * 32;     // this warp's rows (32 * quarter + lane) and columns
        const uint32_t lane_addr = tmem_base + (uint32_t(quarter * 32) << 16) + c0;
        float* colw_s = ctl->colw[warp - 4];
        const float2* colw = reinterpret_cast<const float2*>(colw_s);
        bool ok = true;
        uint32_t acc = 0, parity = 0;
        uint32_t* lam_bits = reinterpret_cast<uint32_t*>(sent_lam);
        // the CTA whose range holds a pair
        auto owner = [&](int pair) {
            const long long x = (long long)(pair + 1) * ctas - 1;
            return x < (1ll << 32) ? int(uint32_t(x) / uint32_t(total)) : int(x / total);
        };
        GramWalk w;
        w.start(ipref, first, count);
        int slab = -1, S = 0, done = 0;                              // of the present slab: sentences, pairs of this range so far
#pragma unroll 1
        while (w.left > 0) {
            // a part of column block J: m pairs from t on
            if (w.slab != slab) { slab = w.slab; S = sent_of(slab); done = 0; }
            const int J = w.J, m = min(J + 1 - w.t, w.left), j0 = J * 128 + c0;
            const size_t base = size_t(slab) * max_sent;
            float* p_slab = parts + size_t(slab) * parts_slab;           // [4 * blocks][max_sent]
            const bool full = (J + 1) * 128 <= S;
            const bool my_col = j0 + lane < S;
            float2 cs[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) cs[k] = make_float2(0.f, 0.f);
            // weights of the columns in row sums (nothing for those that are none of the slab's, which are products of zeros)
            const float wj = !my_col ? 0.f : kPass == 2 ? sc_z[base + j0 + lane] : 1.f;
            __syncwarp();
            colw_s[lane] = wj;
            __syncwarp();
            bool diag = w.t == 0;
            int i = (diag ? J : w.t - 1) * 128 + quarter * 32 + lane;
            float* rows = p_slab + size_t(J * 4 + cg) * max_sent;
#pragma unroll 1
            for (int left = m; left > 0; --left) {
                // of this row in column sums (I < J: all rows are the slab's)
                const float wi = diag && i >= S ? 0.f : kPass == 2 ? sc_z[base + i] : 1.f;
                if (ok) {
                    // (inline: a call would spill the sums)
                    bool r = mbar_try_wait(&ctl->tfull[acc], parity);
                    for (uint32_t n = 0; !r && n < limit; ++n) {
                        if ((n & 63) == 63 && *reinterpret_cast<volatile int*>(&ctl->abort_flag)) break;
                        r = mbar_try_wait(&ctl->tfull[acc], parity);
                    }
                    ok = __all_sync(0xffffffffu, r);
                    if (!ok) {
                        atomicOr(status, SKIPKV_STATUS_COPY_TIMEOUT);
                        *reinterpret_cast<volatile int*>(&ctl->abort_flag) = 1;
                    }
                }
                if (ok) {
                    tc_fence_after();
                    float v[32];
                    tmem_ld32(lane_addr + acc * 128, v);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->tempty[acc]);
                    const bool plain = !diag && full;
                    if (kPass == 1 && !ext.table) {
                        float mx = -INFINITY, m1 = -INFINITY;
                        if (plain) {
#pragma unroll
                            for (int k = 0; k < 32; k += 4) { mx = max3(mx, v[k], v[k + 1]); m1 = max3(m1, v[k + 2], v[k + 3]); }
                        } else {
                            const int from = i - j0, to = S - j0;    // later sentences only
#pragma unroll
                            for (int k = 0; k < 32; ++k)
                                if (k > from && k < to) mx = fmaxf(mx, v[k]);
                        }
                        mx = fmaxf(mx, m1);
                        if (mx > tau) atomicMax(lam_bits + base + i, ordered_bits(mx));
                    }
                    if (diag && quarter == cg) {                     // a sentence and itself
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            if (k == lane) v[k] = -INFINITY;
                    }
                    float2 row = make_float2(0.f, 0.f);
                    const float2 l2 = make_float2(kLog2e, kLog2e), w2 = make_float2(wi, wi);
                    if (kPass == 1 && plain) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const float2 x = __fmul2_rn(make_float2(v[2 * k], v[2 * k + 1]), l2), e = make_float2(ex2f(x.x), ex2f(x.y));
                            row = __fadd2_rn(row, e);
                            cs[k] = __fadd2_rn(cs[k], e);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const float2 x = __fmul2_rn(make_float2(v[2 * k], v[2 * k + 1]), l2), e = make_float2(ex2f(x.x), ex2f(x.y));
                            row = __ffma2_rn(e, colw[k], row);
                            cs[k] = __ffma2_rn(e, w2, cs[k]);
                        }
                    }
                    // (the diagonal pair is symmetric: its column sums are all there is to it)
                    if (!diag) rows[i] = row.x + row.y;
                }
                if (++acc == kGramAcc) { acc = 0; parity ^= 1u; }
                i = diag ? quarter * 32 + lane : i + 128;
                diag = false;
            }
            if (ok) {
                float s[32];
#pragma unroll
                for (int k = 0; k < 16; ++k) { s[2 * k] = cs[k].x; s[2 * k + 1] = cs[k].y; }
                const float sum = col_reduce32(s, lane);
                const int part = w.t == 0 ? 0 : cta - owner(ipref[slab] + J * (J + 1) / 2);
                if (my_col) p_slab[size_t(part * 4 + quarter) * max_sent + j0 + lane] = sum;
            }
            done += m;
            w.advance(ipref, m);
            if (w.slab != slab || w.left == 0) {                     // the range's part of this slab is complete
                __threadfence();
                named_bar_sync(1, 512);
                const int nb = (S + 127) >> 7;
                if (warp == 4 && lane == 0) {
                    const int all = nb * (nb + 1) / 2;
                    const int have = ok ? int(atomicAdd(cnt + slab, uint32_t(done))) + done : 0;
                    ctl->last = have == all;
                    if (have == all) cnt[slab] = 0u;                 // for the next pass or call
                    __threadfence();
                }
                named_bar_sync(1, 512);
                if (*reinterpret_cast<volatile int*>(&ctl->last)) {
                    for (int k = tid - 128; k < S; k += 512) {
                        // the parts of block b's columns, then its rows with the blocks after it
                        const int b = k >> 7, x0 = ipref[slab] + b * (b + 1) / 2, n_part = owner(x0 + b) - owner(x0) + 1;
                        float sum = 0.f;
                        auto add = [&](int from, int to) {
                            const float* x = p_slab + size_t(from) * 4 * max_sent + k;
#pragma unroll 8
                            for (int q = from; q < to; ++q, x += 4 * size_t(max_sent))
                                sum += (__ldcg(x) + __ldcg(x + max_sent)) + (__ldcg(x + 2 * max_sent) + __ldcg(x + 3 * max_sent));
                        };
                        add(0, n_part);
                        add(b + 1, nb);
                        const size_t o = base + k;
                        if (kPass == 1) {
                            sc_z[o] = sum > 0.f ? 1.f / sum : 0.f;
                        } else {
                            const float red = sum / float(S);
                            float lam;
                            if (ext.table) {                         // penalty from the generation-space table through Phi
                                const int g = ext.sent_id[o];
                                lam = (g >= 0 && g < ext.table_len) ? ext.table[size_t(slab / ext.Hk) * ext.table_len + g] : 0.f;
                            } else {
                                const uint32_t u = lam_bits[o];
                                lam = u ? from_ordered_bits(u) : 0.f;
                            }
                            sent_lam[o] = lam;
                            sent_red[o] = red;
                            sent_score[o] = sigma * sent_imp[o] - (1.f - sigma) * red - lam;
                        }
                    }
                }
                named_bar_sync(1, 512);                              // `last` may be written again
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 128 * kGramAcc);
    }
}

// ---------------------------------------------------------------------------------------
// Everything after the sweeps for slabs of at most 128 sentences (caches near a budget of a few thousand tokens): one CTA
// per slab pools its sentences, puts the pooled keys' high and low parts into shared memory as operand tiles, multiplies
// them once, and takes the row sums, the penalties, the redundancy and the scores from the one accumulator, whose
// exponentials stay in registers between the two uses.  Nothing but latency bounds these slabs: the three kernels this
// replaces (pooling and two Gram passes, for any number of sentences) took 22 us for 8 slabs and 28 us for 80, each
// waiting for the one before it to drain.  16 warps, so that all rows' loads are one batch: 22.3 -> 18.2 us a launch (with its
// wait for the sweep) against 8 warps with two.
// ---------------------------------------------------------------------------------------
constexpr int kSmallThreads = 512;
constexpr int kSmallBatch = 8;          // sentences of a warp: their loads are in flight together
struct SmallCtl {
    uint64_t done;
    uint32_t tmem_base;
    alignas(16) float imp[kSmallSent], sum[4][kSmallSent], mx[4][kSmallSent], red[4][kSmallSent], invz[kSmallSent];
};
constexpr size_t kSmallSmem = 1024 + 2 * size_t(kOpBytes) + sizeof(SmallCtl);

__global__ void __launch_bounds__(kSmallThreads)
score_small_kernel(uint32_t* lse_cnt, int Hk, int max_sent, int max_cap, int max_rows, const int32_t* cap, const int32_t* kv_len, const int32_t* sent_off,
                   const int32_t* n_sent, float eps, float sigma, float tau, const float* tok_imp_ws, const float* vsum,
                   float* sent_imp, float* sent_red, float* sent_lam, float* sent_score, LamTable ext, const Header* hdr) {
    extern __shared__ uint8_t small_smem_raw[];
    const uint32_t raw = smem_u32(small_smem_raw);
    uint8_t* hi_t = small_smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint8_t* lo_t = hi_t + kOpBytes;
    SmallCtl* ctl = reinterpret_cast<SmallCtl*>(lo_t + kOpBytes);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slab = blockIdx.x;
    pdl_trigger();
    if (tid == 0) { mbar_init(&ctl->done, 1); mbar_fence_init(); }
    if (warp == 1) tmem_alloc(&ctl->tmem_base, 128);
    pdl_wait();
    if (tid < 2) lse_cnt[tid * gridDim.x + slab] = 0u;   // both counters, for the next call's sweeps
    const int S = min(max(n_sent[slab], 0), max_sent), N = min(max(kv_len[slab], 0), min(cap[slab / Hk], max_rows));
    const int32_t* so = sent_off + size_t(slab) * (max_sent + 1);
    const float* ti_p = tok_imp_ws + size_t(slab) * max_cap;
    // ---- pooling: kSmallBatch rows per warp; rows past the last sentence are zeros
    {
        const int i0 = warp * kSmallBatch, cnt = min(kSmallBatch, S - i0);
        const int off = lane <= cnt ? so[i0 + lane] : 0;
        float4 v[kSmallBatch];
#pragma unroll
        for (int u = 0; u < kSmallBatch; ++u)
            v[u] = u < cnt ? reinterpret_cast<const float4*>(vsum + (size_t(slab) * max_sent + i0 + u) * kHeadDim)[lane]
                           : make_float4(0.f, 0.f, 0.f, 0.f);
        float ti[kSmallBatch];
        int beg[kSmallBatch], end[kSmallBatch];
#pragma unroll
        for (int u = 0; u < kSmallBatch; ++u) {
            beg[u] = max(__shfl_sync(0xffffffffu, off, u), 0);
            end[u] = min(__shfl_sync(0xffffffffu, off, u + 1), N);
            if (u >= cnt) end[u] = beg[u];
            const int t = beg[u] + lane;                 // most sentences have at most 64 tokens: two loads, all in flight
            ti[u] = t < end[u] ? ti_p[t] : 0.f;
            if (t + 32 < end[u]) ti[u] += ti_p[t + 32];
        }
#pragma unroll
        for (int u = 0; u < kSmallBatch; ++u)
            for (int t = beg[u] + lane + 64; t < end[u]; t += 32) ti[u] += ti_p[t];
#pragma unroll
        for (int u = 0; u < kSmallBatch; ++u) {
            const int n = end[u] - beg[u], r = i0 + u;
            const float inv_len = n > 0 ? 1.f / float(n) : 0.f;
            float4 x = n > 0 ? v[u] : make_float4(0.f, 0.f, 0.f, 0.f);
            x.x *= inv_len; x.y *= inv_len; x.z *= inv_len; x.w *= inv_len;
            float nn = x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w, ts = ti[u];
#pragma unroll
            for (int d = 16; d; d >>= 1) {
                nn += __shfl_xor_sync(0xffffffffu, nn, d);
                ts += __shfl_xor_sync(0xffffffffu, ts, d);
            }
            const float inv = 1.f / (sqrtf(nn) + eps);
            const float y[4] = {x.x * inv, x.y * inv, x.z * inv, x.w * inv};
            uint32_t hi[4], lo[4];                       // bf16 bit patterns
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const __nv_bfloat16 h = __float2bfloat16_rn(y[c]);
                hi[c] = __bfloat16_as_ushort(h);
                lo[c] = __bfloat16_as_ushort(__float2bfloat16_rn(y[c] - __bfloat162float(h)));
            }
            // channels 4 lane .. 4 lane + 3 of row r, as a tiled copy with the 128-byte swizzle would place them
            const int at = (lane >> 4) * kOpHalfBytes + r * 128 + ((((lane & 15) >> 1) ^ (r & 7)) << 4) + (lane & 1) * 8;
            *reinterpret_cast<uint2*>(hi_t + at) = make_uint2(hi[0] | (hi[1] << 16), hi[2] | (hi[3] << 16));
            *reinterpret_cast<uint2*>(lo_t + at) = make_uint2(lo[0] | (lo[1] << 16), lo[2] | (lo[3] << 16));
            if (lane == 0 && u < cnt) {
                const float imp = n > 0 ? ts * inv_len : 0.f;
                ctl->imp[r] = imp;
                sent_imp[size_t(slab) * max_sent + r] = imp;
            }
        }
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (warp == 0) {
        const uint32_t a = smem_u32(hi_t), b = smem_u32(lo_t), leader = elect_leader();
        umma_tile_128x128x128(tmem_base, a, a, false, leader);
        umma_tile_128x128x128(tmem_base, a, b, true, leader);
        umma_tile_128x128x128(tmem_base, b, a, true, leader);
        umma_commit(&ctl->done, leader);
    }
    const bool ok = mbar_wait(&ctl->done, 0u, load_wait_limit(hdr));
    if (!ok) {                                           // the outputs are skipped, but the product retires before it is read or released
        if (lane == 0) atomicOr(const_cast<uint32_t*>(&hdr->status), SKIPKV_STATUS_COPY_TIMEOUT);
        mbar_wait(&ctl->done, 0u, kRetirePolls);
    }
    __syncwarp();
    tc_fence_after();
    // ---- thread: row i, 32 columns; four warps share a row
    const int part = warp >> 2, i = (warp & 3) * 32 + lane, c0 = part * 32;
    float e[32];
    float sum = 0.f, mx = -INFINITY;
    if (c0 < S) {                                        // (the same for the whole warp)
        tmem_ld32(tmem_base + (uint32_t((warp & 3) * 32) << 16) + c0, e);
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) {
            const int j = c0 + jj;
            const bool on = j < S && j != i;
            if (on && j > i) mx = fmaxf(mx, e[jj]);
            e[jj] = on ? ex2f(e[jj] * kLog2e) : 0.f;
            sum += e[jj];
        }
    } else {
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) e[jj] = 0.f;
    }
    ctl->sum[part][i] = sum;
    ctl->mx[part][i] = mx;
    tc_fence_before();
    __syncthreads();
    if (part == 0) {
        const float z = (sum + ctl->sum[1][i]) + (ctl->sum[2][i] + ctl->sum[3][i]);
        ctl->invz[i] = (i < S && z > 0.f) ? 1.f / z : 0.f;
    }
    __syncthreads();
    float red = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 iz = *reinterpret_cast<const float4*>(&ctl->invz[c0 + q * 4]);
        red = fmaf(e[q * 4], iz.x, red);
        red = fmaf(e[q * 4 + 1], iz.y, red);
        red = fmaf(e[q * 4 + 2], iz.z, red);
        red = fmaf(e[q * 4 + 3], iz.w, red);
    }
    ctl->red[part][i] = red;
    __syncthreads();
    if (part == 0 && i < S && ok) {
        const size_t o = size_t(slab) * max_sent + i;
        float lam = fmaxf(fmaxf(mx, ctl->mx[1][i]), fmaxf(ctl->mx[2][i], ctl->mx[3][i]));
        if (ext.table) {                                 // penalty from the generation-space table through Phi
            const int g = ext.sent_id[o];
            lam = (g >= 0 && g < ext.table_len) ? ext.table[size_t(slab / Hk) * ext.table_len + g] : 0.f;
        } else {
            lam = (lam > tau) ? lam : 0.f;
        }
        red = ((red + ctl->red[1][i]) + (ctl->red[2][i] + ctl->red[3][i])) / float(S);
        sent_lam[o] = lam;
        sent_red[o] = red;
        sent_score[o] = sigma * ctl->imp[i] - (1.f - sigma) * red - lam;
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 128);
    }
}

}  // namespace skipkv

using namespace skipkv;

static int score_impl(const skipkv_shape* shape, const skipkv_params* params, const void* K, const void* q_win,
                      const int32_t* kv_len, const int32_t* sent_off, const int32_t* n_sent, float* tok_imp,
                      float* sent_imp, float* sent_red, float* sent_lam, float* sent_score, LamTable ext, void* ws,
                      void* stream, const int32_t* block_table = nullptr, int max_pages = 0) {
    if (int rc = check_shape(shape)) return rc;
    if (!params || !K || !q_win || !kv_len || !sent_off || !n_sent || !sent_imp || !sent_red || !sent_lam || !sent_score)
        return SKIPKV_ERR_INVALID_ARG;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return SKIPKV_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(K) & 15) || (reinterpret_cast<uintptr_t>(q_win) & 15)) return SKIPKV_ERR_INVALID_ARG;
    if (shape->max_sent <= 0) return SKIPKV_OK;
    const WsLayout L = make_layout(*shape);
    uint8_t* w = static_cast<uint8_t*>(ws);
    uint32_t* status = &reinterpret_cast<Header*>(w + L.header)->status;
    float* sc_tok = reinterpret_cast<float*>(w + L.sc_tokimp);
    float* vsum = reinterpret_cast<float*>(w + L.sc_vsum);
    __nv_bfloat16* vbar_hi = reinterpret_cast<__nv_bfloat16*>(w + L.sc_vbar_hi);
    __nv_bfloat16* vbar_lo = reinterpret_cast<__nv_bfloat16*>(w + L.sc_vbar_lo);
    float* sc_z = reinterpret_cast<float*>(w + L.sc_z);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int Hq = shape->n_q_heads, Hk = shape->n_kv_heads, n = L.group;

    CUtensorMap mapK, mapQ, mapHi{}, mapLo{};
    if (int rc = tmap_rows(&mapK, K, uint64_t(shape->total_rows), 128)) return rc;
    if (int rc = tmap_groups(&mapQ, q_win, uint64_t(shape->batch) * Hq, uint32_t(shape->window), uint32_t(L.sc_wb), uint32_t(n)))
        return rc;
    if (shape->max_sent > kSmallSent) {
        if (int rc = tmap_groups(&mapHi, vbar_hi, uint64_t(L.slabs), uint32_t(shape->max_sent), 128, 1)) return rc;
        if (int rc = tmap_groups(&mapLo, vbar_lo, uint64_t(L.slabs), uint32_t(shape->max_sent), 128, 1)) return rc;
    }

    SweepArgs a{};
    a.Hq = Hq; a.Hk = Hk; a.window = shape->window; a.n_slabs = L.slabs; a.max_cap = shape->max_cap;
    a.max_sent = shape->max_sent;
    a.WB = L.sc_wb; a.RB = L.sc_rb; a.N = L.sc_wb * n; a.R = a.RB * a.N; a.RA = L.sc_ra;
    a.slab_off = shape->slab_off; a.cap = shape->cap; a.kv_len = kv_len; a.sent_off = sent_off; a.n_sent = n_sent;
    a.rec = reinterpret_cast<float2*>(w + L.sc_part); a.lse_cnt = reinterpret_cast<uint32_t*>(w + L.sc_cnt); a.sum_cnt = a.lse_cnt + L.slabs;
    a.tok_imp_user = tok_imp; a.tok_imp_ws = sc_tok; a.vsum = vsum; a.status = status;
    a.pool_a = a.RA == 1;                            // see the head of the sweeps
    a.hdr = reinterpret_cast<const Header*>(w + L.header);
    a.block_table = block_table; a.max_pages = max_pages;
    const size_t max_smem = 227 * 1024;
    size_t fixed = 1024 + size_t(a.R) * kRowBytes + 2 * kIndBytes + 128 * kExtRow + sweep_ext_bytes(a.R, a.RA) +
                   sizeof(SweepCtl) + size_t(a.RB - 1) * 4 * 128 * 4;
    // The table of slabs (8 bytes each) goes into shared memory as long as one tile stage fits beside it: all but windows of some hundred
    // query rows with hundreds of slabs and more.  Of 512 rows, one head x 512 positions leaves room for 948 slabs, four heads x 128 for 4000 (six heads x 84,
    // padded to 576 rows, 436); without the other form the call would end there.
    const size_t table_bytes = size_t(2 * L.slabs + 1) * 4;
    const bool in_global = fixed + table_bytes + kOpBytes > max_smem;
    if (in_global) a.table = reinterpret_cast<int*>(w + L.slab_table);
    else fixed += table_bytes;
    const size_t gsmem = gram_smem_bytes(L.slabs);
    if (shape->max_sent > kSmallSent && gsmem > max_smem) {          // (before anything is enqueued)
        set_error_text("skipkv_score: more than 128 sentences per slab and batch * n_kv_heads too large for the shared-memory table of the Gram kernels");
        return SKIPKV_ERR_UNSUPPORTED;
    }
    // Four indicator matrices in flight (two more than counted above) wherever that leaves two tile stages: with two a matrix waits for the
    // product two tiles back, and pass A took 1.15 us a tile instead of 0.85 (80 slabs of 16K to 32K rows).
    a.ind_log = fixed + 2 * kIndBytes + 2 * kOpBytes <= max_smem ? 2 : 1;
    if (a.ind_log == 2) fixed += 2 * kIndBytes;
    a.stages = int((max_smem - fixed) / kOpBytes);
    if (a.stages > kStagesMax) a.stages = kStagesMax;
    int grid = num_sms();
    if (grid > L.dec_max_ctas) grid = L.dec_max_ctas;
    // Cooperative: the CTAs wait for one another between the passes, so they have to be resident together whatever else
    // runs on the GPU.  Where the context may use fewer SMs than the device has, a smaller grid does.
    cudaError_t le = cudaErrorCooperativeLaunchTooLarge;
    if (in_global) SKIPKV_CUDA(launch_dependent(sweep_table_kernel, dim3(1), dim3(1024), 0, st, a));
    const auto sweep = L.sc_wb == 32 ? (in_global ? score_sweep_kernel<32, true> : score_sweep_kernel<32, false>)
                                     : (in_global ? score_sweep_kernel<16, true> : score_sweep_kernel<16, false>);
    for (; grid >= 1 && le == cudaErrorCooperativeLaunchTooLarge; grid /= 2) {
        le = launch_dependent<true>(sweep, dim3(grid), dim3(kSweepThreads), fixed + size_t(a.stages) * kOpBytes, st, mapK, mapQ, a);
        if (le == cudaErrorCooperativeLaunchTooLarge) (void)cudaGetLastError();
        else break;
    }
    SKIPKV_CUDA(le);
    const int max_rows = block_table ? max_pages * 128 : 0x7fffffff;          // rows the sweeps look at
    // one tile of sentences per slab: one kernel instead of three, with the operands in shared memory throughout
    if (shape->max_sent <= kSmallSent) {
        SKIPKV_CUDA(launch_dependent(score_small_kernel, dim3(L.slabs), dim3(kSmallThreads), kSmallSmem, st, a.lse_cnt, Hk, int(shape->max_sent),
                                     int(shape->max_cap), max_rows, shape->cap, kv_len, sent_off, n_sent, params->eps, params->sigma,
                                     params->tau, static_cast<const float*>(sc_tok), static_cast<const float*>(vsum), sent_imp,
                                     sent_red, sent_lam, sent_score, ext, reinterpret_cast<const Header*>(w + L.header)));
        return SKIPKV_OK;
    }
    {
        dim3 pgrid(unsigned(shape->max_sent + 8 * kPoolRows - 1) / (8 * kPoolRows), L.slabs);
        SKIPKV_CUDA(launch_dependent(score_pool_kernel, pgrid, dim3(256), 0, st, a.lse_cnt, Hk, shape->max_sent, shape->max_cap, max_rows,
                                     shape->cap, kv_len, sent_off, n_sent, params->eps, sc_tok, vsum, sent_imp, vbar_hi,
                                     vbar_lo, sent_lam));
    }
    {
        const long long nb = (shape->max_sent + 127) / 128, max_items = L.slabs * (nb * (nb + 1) / 2);
        const int ggrid = int(max_items < (long long)grid ? max_items : (long long)grid);
        SKIPKV_CUDA(launch_dependent(score_gram_kernel<1>, dim3(ggrid), dim3(kGramThreads), gsmem, st, mapHi, mapLo, L.slabs,
                                     shape->max_sent, n_sent, params->sigma, params->tau, sc_z, sent_imp, sent_red, sent_lam,
                                     sent_score, vsum, L.sc_vsum_slab, a.lse_cnt, ext, reinterpret_cast<const Header*>(w + L.header)));
        SKIPKV_CUDA(launch_dependent(score_gram_kernel<2>, dim3(ggrid), dim3(kGramThreads), gsmem, st, mapHi, mapLo, L.slabs,
                                     shape->max_sent, n_sent, params->sigma, params->tau, sc_z, sent_imp, sent_red, sent_lam,
                                     sent_score, vsum, L.sc_vsum_slab, a.lse_cnt, ext, reinterpret_cast<const Header*>(w + L.header)));
    }
    return SKIPKV_OK;
}

extern "C" int skipkv_score(const skipkv_shape* shape, const skipkv_params* params, const void* K, const void* q_win,
                            const int32_t* kv_len, const int32_t* sent_off, const int32_t* n_sent, float* tok_imp,
                            float* sent_imp, float* sent_red, float* sent_lam, float* sent_score, void* ws,
                            void* stream) {
    return score_impl(shape, params, K, q_win, kv_len, sent_off, n_sent, tok_imp, sent_imp, sent_red, sent_lam,
                      sent_score, LamTable{nullptr, nullptr, 0, 1}, ws, stream);
}

extern "C" int skipkv_score_table(const skipkv_shape* shape, const skipkv_params* params, const void* K,
                                  const void* q_win, const int32_t* kv_len, const int32_t* sent_off,
                                  const int32_t* sent_id, const int32_t* n_sent, const float* lam_table,
                                  int32_t table_len, float* tok_imp, float* sent_imp, float* sent_red, float* sent_lam,
                                  float* sent_score, void* ws, void* stream) {
    if (!sent_id || !lam_table || table_len <= 0) return SKIPKV_ERR_INVALID_ARG;
    if (int rc = check_shape(shape)) return rc;
    return score_impl(shape, params, K, q_win, kv_len, sent_off, n_sent, tok_imp, sent_imp, sent_red, sent_lam,
                      sent_score, LamTable{lam_table, sent_id, table_len, shape->n_kv_heads}, ws, stream);
}

extern "C" int skipkv_score_paged(const skipkv_shape* shape, const skipkv_params* params, const void* K_pages,
                                  const int32_t* block_table, int32_t max_pages, const void* q_win, const int32_t* kv_len,
                                  const int32_t* sent_off, const int32_t* n_sent, float* tok_imp, float* sent_imp,
                                  float* sent_red, float* sent_lam, float* sent_score, void* ws, void* stream) {
    if (!block_table || max_pages <= 0) return SKIPKV_ERR_INVALID_ARG;
    if (int rc = check_shape(shape)) return rc;
    if (int64_t(max_pages) * 128 > int64_t(shape->max_cap) + 127) return SKIPKV_ERR_INVALID_ARG;   // the workspace is sized by max_cap
    return score_impl(shape, params, K_pages, q_win, kv_len, sent_off, n_sent, tok_imp, sent_imp, sent_red, sent_lam,
                      sent_score, LamTable{nullptr, nullptr, 0, 1}, ws, stream, block_table, max_pages);
}
