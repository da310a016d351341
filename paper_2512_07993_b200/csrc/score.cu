// skipkv_score: sentence scores per (sequence, KV head) slab (paper Section 4.1).
//
//   sweeps    (one launch) pass A: log-sum-exp of every window-query row over the slab's tokens
//             (tensor cores: logits = Q_rows x K_tile^T, one thread per query row);
//             pass B: tok_imp[t] = (1/alpha) sum_w max_q 2^(s_q[w][t] - lse_q[w])   (max before exp: exp is monotone)
//             (tensor cores: logits - (lse - e) = [K_tile, 1] x [Q_block, e - lse]^T, one thread per token; e: see lse_shift), and in the same pass
//             the per-sentence sums of the key rows as a second product on the tile already in shared
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
// group's query rows) into shared memory, two threads in two warps issue tcgen05.mma in turn into a ring of tensor-memory accumulators,
// epilogue warpgroups take the products round-robin (four in pass A, three in pass B), and in pass B one more warpgroup writes the 0/1
// matrices of the pooling product and reads out the pooled sums while one thread of a further warp issues
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
//   pass B   importance of every token and the per-sentence key sums
// Between the two it waits, slab by slab, until every CTA that shares the slab has left its record (a counter of tiles);
// nobody waits for anything but pass A of CTAs that are all resident (one per SM), and the waits are bounded anyway.
// As two launches the second started its first tile 6 us after the first had drained.  Pass A runs backwards through the
// range, so that pass B finds the tiles read last in L2 -- or, where the range fits into the ring, still in shared memory.
// ---------------------------------------------------------------------------------------
constexpr int kStagesMax = 6;
constexpr int kAGroups = 4;             // pass A: epilogue warpgroups = accumulators of 128 columns
constexpr int kBGroups = 3;             // pass B: epilogue warpgroups = accumulators of up to 160 columns
constexpr int kBAccCols = 160;
constexpr int kIndRing = 2;             // indicator matrices in flight (the pooled sums have two accumulators of their own)
constexpr int kIndSlots = 16;           // sentence slots of one indicator matrix
constexpr int kIndBytes = kIndSlots * 128 * 2;   // [16 slots][128 tokens] bf16 as two 64-token halves, 128-byte swizzle
constexpr uint32_t kPoolCol = kBGroups * kBAccCols;   // tensor-memory column of the first pooled-sum accumulator (16 columns each)
constexpr int kPoolWarps = 4;
constexpr int kSweepThreads = (2 + 4 * kAGroups + 2) * 32;    // TMA warp, MMA warp, 16 epilogue warps, issuer of the pooling products, second MMA warp
constexpr int kMaxBlocksA = 5;          // blocks of 128 query rows
constexpr int kExtRow = 32;             // bytes of a row of the extra K step (16 bf16)
constexpr float kLog2e = 1.4426950408889634f;

struct SweepCtl {                       // barriers and small shared state, after the tile buffers
    uint64_t full[kStagesMax], empty[kStagesMax];
    uint64_t qfull, qempty;
    // accumulator i belongs to epilogue warpgroup i (a product of a tile and a block of query rows goes to product number % groups)
    uint64_t tfull_a[kAGroups], tempty_a[kAGroups], tfull_b[kBGroups];
    uint64_t tempty_b[2 * kBGroups];    // by product number: a product waits for the one kBGroups before it, which is the other MMA warp's, and
                                        // with twice as many barriers as accumulators each has one waiter that sees all its phases
    uint64_t tokfull[4];                // pass B, several blocks per tile: the shares of a tile's tokens from all blocks but the last
    uint64_t extfull, extempty;         // pass B: the rows' -lse as operand columns
    // ring of indicator matrices: written by the four pooling warps -> multiplied by their issuer -> read out by the pooling warps
    uint64_t ifull[kIndRing], iempty[kIndRing];
    uint64_t pfull[2];                  // the last product of a run of tiles into accumulator i has completed
    uint64_t retired[3];                // every product of the MMA warps (0, 1) / the pooling issuer (2) has completed
    uint32_t tmem_base;
    int abort_flag;
    int ind_flags[kIndRing];            // 1: the tile has another matrix after this one, 2: joins the open run, 4: closes a run
    uint32_t wsum[32];
};

struct SweepArgs {
    int Hq, Hk, window, n_slabs, max_cap, max_sent, stages;
    int WB, RB, N, R, RA;               // window positions per block of pass B, its blocks, their rows N = WB * n; all rows R = RB * N; blocks of pass A
    const int64_t* slab_off;
    const int32_t* cap;
    const int32_t* kv_len;
    const int32_t* sent_off;
    const int32_t* n_sent;
    float2* rec;                        // [cta + slab][RA * 128] (reference, sum) of a CTA's part of a slab
    uint32_t* lse_cnt;                  // [slabs] tiles whose records are written; zero at the start
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
// Bounded wait of one thread until *p reaches `want`; gives up like role_wait.
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
template <bool kMasked>
__device__ __forceinline__ void lse_fold(uint32_t taddr, int valid, float scale, float& m, float& l) {
    const int nch = kMasked ? (valid + 31) >> 5 : 4;
#pragma unroll 1
    for (int ch = 0; ch < nch; ++ch) {
        float v[32];
        tmem_ld32(taddr + ch * 32, v);
        if (kMasked && ch * 32 + 32 > valid) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (ch * 32 + j >= valid) v[j] = -INFINITY;
        }
        auto chunk_max = [&]() {
            float c0 = fmaxf(v[0], v[1]), c1 = fmaxf(v[2], v[3]);
#pragma unroll
            for (int j = 4; j < 32; j += 4) { c0 = max3(c0, v[j], v[j + 1]); c1 = max3(c1, v[j + 2], v[j + 3]); }
            return fmaxf(c0, c1) * scale;
        };
        auto chunk_sum = [&]() {
            float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
            const float neg = -m;
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                s0 += ex2f(fmaf(v[j + 0], scale, neg));
                s1 += ex2f(fmaf(v[j + 1], scale, neg));
                s2 += ex2f(fmaf(v[j + 2], scale, neg));
                s3 += ex2f(fmaf(v[j + 3], scale, neg));
            }
            return (s0 + s1) + (s2 + s3);
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

// ---- pass B: pooled key sums on the tensor cores
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
// One 16-byte piece of an indicator matrix: tokens 8c .. 8c + 7 of slot row j; ones (bf16 1.0) for the tokens
// [lo, hi), zeros elsewhere.
__device__ __forceinline__ void indicator_piece(uint8_t* ind, int j, int c, int lo, int hi) {
    const int b0 = min(max(lo - 8 * c, 0), 8), b1 = min(max(hi - 8 * c, 0), 8);
    const uint32_t m8 = b1 > b0 ? (((1u << b1) - 1u) & ~((1u << b0) - 1u)) : 0u;
    uint4 val;
    val.x = (m8 & 1u) * 0x3F80u + ((m8 >> 1) & 1u) * 0x3F800000u;
    val.y = ((m8 >> 2) & 1u) * 0x3F80u + ((m8 >> 3) & 1u) * 0x3F800000u;
    val.z = ((m8 >> 4) & 1u) * 0x3F80u + ((m8 >> 5) & 1u) * 0x3F800000u;
    val.w = ((m8 >> 6) & 1u) * 0x3F80u + ((m8 >> 7) & 1u) * 0x3F800000u;
    *reinterpret_cast<uint4*>(ind + (c >> 3) * (kIndBytes / 2) + j * 128 + (((c & 7) ^ (j & 7)) << 4)) = val;
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
    uint8_t* indb = tiles + size_t(a.stages) * kOpBytes;                         // pass B: the indicator matrices
    uint8_t* onesb = indb + kIndRing * kIndBytes;                                // pass B: the keys' side of the extra K step
    uint8_t* extb = onesb + 128 * kExtRow;                                       // pass B: the queries' side; pass A: [4 groups][RA * 128] (m, l)
    SweepCtl* ctl = reinterpret_cast<SweepCtl*>(extb + size_t(a.RA) * 128 * kExtRow);
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
        for (int s = 0; s < kStagesMax; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], a.RB > 1 ? 3 : 2); }
        mbar_init(&ctl->qfull, 1);
        mbar_init(&ctl->qempty, 2);
        for (int g = 0; g < kAGroups; ++g) { mbar_init(&ctl->tfull_a[g], 1); mbar_init(&ctl->tempty_a[g], 4); }
        for (int g = 0; g < kBGroups; ++g) { mbar_init(&ctl->tfull_b[g], 1); mbar_init(&ctl->tempty_b[g], 4); mbar_init(&ctl->tempty_b[kBGroups + g], 4); }
        for (int i = 0; i < 4; ++i) mbar_init(&ctl->tokfull[i], a.RB > 1 ? 4 * (a.RB - 1) : 1);
        mbar_init(&ctl->extfull, 4);
        mbar_init(&ctl->extempty, 2);
        for (int i = 0; i < kIndRing; ++i) { mbar_init(&ctl->ifull[i], kPoolWarps); mbar_init(&ctl->iempty[i], 1); }
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
    const bool resident = ntl <= a.stages;               // the range fits into the ring: pass B reads it where pass A left it
    const float scale = kLog2e * rsqrtf(float(kHeadDim));
    const int n = a.Hq / Hk;
    const uint32_t ext_smem = smem_u32(extb);
    // Pass A, last block of at most 64 rows: on every second tile its rows take the upper tensor-memory lanes, so that the
    // exponentials spread over all four schedulers.  (Which tiles an epilogue group gets its last block from has one parity
    // for each group when there are 2, 3 or 5 blocks.)
    const bool can_shift = a.RA > 1 && a.RA != 4 && a.R - (a.RA - 1) * 128 <= 64;
    auto shifted = [&](int i) { return can_shift && (i & 1); };

    if (ntl > 0) {
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            // what depends on the slab only is kept in registers: between "stage free" and the next copy's issue nothing
            // waits on shared or global memory
            int stage = 0;
            uint32_t lap = 0, qlap = 0;
            bool ok = true;
            auto load_q = [&](int slab) {
                if (qlap > 0) ok = role_wait(&ctl->qempty, (qlap - 1) & 1u, limit, &ctl->abort_flag, a.status);
                if (!ok) return;
                const int b = slab / Hk, h = slab % Hk;
                mbar_expect_tx(&ctl->qfull, uint32_t(a.R) * kRowBytes);
                for (int k = 0; k < a.RB; ++k)
                    for (int half = 0; half < 2; ++half)
                        tma_load_3d(qbuf + size_t(half) * q_half + size_t(k) * a.N * 128, &mapQ, half * 64, k * kWB, b * a.Hq + h * n, &ctl->qfull);
                ++qlap;
            };
            auto load_tile = [&](int slab, int j, int row0) {
                const int row = a.block_table ? max(a.block_table[size_t(slab) * a.max_pages + j], 0) * 128 : row0 + j * 128;
                if (lap > 0) ok = role_wait(&ctl->empty[stage], (lap - 1) & 1u, limit, &ctl->abort_flag, a.status);
                if (!ok) return;
                uint8_t* dst = tiles + size_t(stage) * kOpBytes;
                mbar_expect_tx(&ctl->full[stage], kOpBytes);
                tma_load_2d(dst, &mapK, 0, row, &ctl->full[stage]);
                tma_load_2d(dst + kOpHalfBytes, &mapK, 64, row, &ctl->full[stage]);
                if (++stage == a.stages) { stage = 0; ++lap; }
            };
            for (int pass = 0; pass < 2 && ok; ++pass) {
                const int t_first = pass == 0 && !resident ? t_end - 1 : t_begin;
                int slab = slab_of(t_first), lo = 0, hi = 0, row0 = 0;          // tiles [lo, hi) belong to the slab
                for (int i = 0; i < ntl && ok; ++i) {
                    const int t = pass == 0 && !resident ? t_end - 1 - i : t_begin + i;
                    if (i == 0 || t >= hi || t < lo) {
                        while (pref[slab + 1] <= t) ++slab;
                        while (pref[slab] > t) --slab;
                        lo = pref[slab]; hi = pref[slab + 1];
                        row0 = rowb[slab];
                        load_q(slab);
                        if (!ok) break;
                    }
                    if (pass == 0 || !resident) load_tile(slab, t - lo, row0);
                }
            }
            // Whoever gave up: this warp stays until its copies have landed and the issuers' products have completed, so that the CTA gives
            // back shared and tensor memory with nothing in flight.  Stage s was loaded lap (+ 1) times.
            for (int s = 0; s < a.stages; ++s) {
                const uint32_t loads = lap + (s < stage ? 1u : 0u);
                if (loads) mbar_wait(&ctl->full[s], (loads - 1) & 1u, kRetirePolls);
            }
            if (qlap) mbar_wait(&ctl->qfull, (qlap - 1) & 1u, kRetirePolls);
            for (int s = 0; s < 3; ++s) mbar_wait(&ctl->retired[s], 0u, kRetirePolls);
        }
    } else if (warp == 1 || warp == 19) {
        // ------------------------------------------------------------------ MMA warps
        // Two of them take the products in turn.  An issue blocks until the tensor core has taken the product, and a look
        // at a barrier in between (115 cycles and more) leaves it idle; with two issuers one waits while the other's
        // product runs (measured without epilogue: 817 against 579 cycles per 128 x 128 x 128 product, 512 the least).
        const int mine = warp == 1 ? 0 : 1;
        const uint32_t leader = elect_leader();
        bool ok = true;
        uint32_t qlap = 0;
        const uint32_t q0 = smem_u32(qbuf);
        {
            int stage = 0, it = 0, slab = slab_of(resident ? t_begin : t_end - 1), lo = 0, hi = 0;
            uint32_t lap = 0;
            const int n_empty = a.RB > 1 ? 3 : 2;        // arrivals that free a stage
            for (int i = 0; i < ntl && ok; ++i) {
                const int t = resident ? t_begin + i : t_end - 1 - i;
                if (i == 0 || t >= hi || t < lo) {
                    while (pref[slab + 1] <= t) ++slab;
                    while (pref[slab] > t) --slab;
                    lo = pref[slab]; hi = pref[slab + 1];
                    ok = warp_wait(&ctl->qfull, qlap & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    ++qlap;
                }
                // (both warps follow every tile's arrival, so that they see each phase of a stage's barrier)
                ok = warp_wait(&ctl->full[stage], lap & 1u, limit, &ctl->abort_flag, a.status);
                bool here = false;                       // this warp has a product of the tile
                for (int k = 0; k < a.RA && ok; ++k, ++it) {
                    if ((it & 1) != mine) continue;
                    here = true;
                    const int buf = it & (kAGroups - 1), use = it / kAGroups;
                    if (use > 0) ok = warp_wait(&ctl->tempty_a[buf], uint32_t(use - 1) & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    tc_fence_after();
                    const int r = k + 1 == a.RA && shifted(i) ? a.R - 128 : k * 128;       // first query row
                    umma_tile(tmem_base + buf * 128, q0 + uint32_t(r) * 128u, q_half, smem_u32(tiles + size_t(stage) * kOpBytes),
                              kOpHalfBytes, kIdescBf16M128N128, leader);
                    umma_commit(&ctl->tfull_a[buf], leader);
                }
                const int t_next = resident ? t + 1 : t - 1;
                if (i + 1 == ntl || t_next >= hi || t_next < lo) umma_commit(&ctl->qempty, leader);
                if (!resident && here) {                 // one warp: all arrivals; two: the second one of the tile makes up the number
                    const int c = a.RA == 1 ? n_empty : (((it - 1) & 1) == mine ? n_empty - 1 : 1);
                    for (int e = 0; e < c; ++e) umma_commit(&ctl->empty[stage], leader);
                }
                if (++stage == a.stages) { stage = 0; ++lap; }
            }
        }
        __syncwarp();
        tc_fence_before();
        named_bar_sync(1, kSweepThreads - 32);           // every accumulator of pass A has been read
        tc_fence_after();
        if (ok) {
            int it = 0, slab = slab_of(t_begin), hi = 0, stage = resident ? 0 : ntl % a.stages;
            uint32_t elap = 0, lap = resident ? 0u : uint32_t(ntl / a.stages);
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t(a.N) >> 3) << 17) | ((128u >> 4) << 24);
            const uint64_t d_ones = umma_desc_sw32(smem_u32(onesb));
            for (int i = 0; i < ntl && ok; ++i) {
                const int t = t_begin + i;
                if (i == 0 || t >= hi) {
                    while (pref[slab + 1] <= t) ++slab;
                    hi = pref[slab + 1];
                    ok = warp_wait(&ctl->qfull, qlap & 1u, limit, &ctl->abort_flag, a.status) &&
                         warp_wait(&ctl->extfull, elap & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    ++qlap; ++elap;
                }
                ok = warp_wait(&ctl->full[stage], lap & 1u, limit, &ctl->abort_flag, a.status);
                bool here = false;
                for (int k = 0; k < a.RB && ok; ++k, ++it) {
                    if ((it & 1) != mine) continue;
                    here = true;
                    const int buf = it % kBGroups, before = it - kBGroups;
                    if (before >= 0) ok = warp_wait(&ctl->tempty_b[before % (2 * kBGroups)], uint32_t(before / (2 * kBGroups)) & 1u, limit, &ctl->abort_flag, a.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d = tmem_base + buf * kBAccCols;
                    umma_tile(d, smem_u32(tiles + size_t(stage) * kOpBytes), kOpHalfBytes, q0 + uint32_t(k * a.N) * 128u, q_half, idesc, leader);
                    umma_bf16(d, d_ones, umma_desc_sw32(ext_smem + uint32_t(k * a.N) * kExtRow), idesc, 1u, leader);      // - lse
                    umma_commit(&ctl->tfull_b[buf], leader);
                }
                if (i + 1 == ntl || hi <= t + 1) { umma_commit(&ctl->qempty, leader); umma_commit(&ctl->extempty, leader); }
                if (here) umma_commit(&ctl->empty[stage], leader);
                if (++stage == a.stages) { stage = 0; ++lap; }
            }
        }
        umma_commit(&ctl->retired[mine], leader);
    } else {
        // ------------------------------------------------------------------ pass A: epilogue warpgroups (and the clearing warp)
        const int quarter = warp & 3;                        // tensor-memory lanes this warp may read
        bool ok = true;
        {
            const int g = (warp - 2) >> 2;                   // warpgroup (warp 18: 4, clears the key sums)
            const int row = quarter * 32 + lane;
            const uint32_t lane_addr = tmem_base + (uint32_t(quarter * 32) << 16) + g * 128;
            float2* part = reinterpret_cast<float2*>(extb);  // [group][RA * 128]
            const bool g_shifted = can_shift && (a.RA == 2 ? g == 3 : (g & 1) != 0);
            const int rem = a.R - (a.RA - 1) * 128;          // rows of the last block
            int it = g, ti = g / a.RA, tk = g - ti * a.RA;   // this group's next product: its number, tile (in the order of the pass) and block
            int slab = slab_of(resident ? t_begin : t_end - 1);
            for (int done = 0; done < ntl;) {
                // one segment: the tiles of a slab that this CTA has
                const int t_cur = resident ? t_begin + done : t_end - 1 - done;
                while (pref[slab + 1] <= t_cur) ++slab;
                while (pref[slab] > t_cur) --slab;
                const int lo = max(pref[slab], t_begin), hi = min(pref[slab + 1], t_end), seg_end = done + (hi - lo);
                const int fc = owner(pref[slab]), lc = owner(pref[slab + 1] - 1);
                if (g < kAGroups) {
                    const int N = live(slab);
                    float m[kMaxBlocksA], l[kMaxBlocksA];
#pragma unroll
                    for (int k = 0; k < kMaxBlocksA; ++k) { m[k] = -INFINITY; l[k] = 0.f; }
                    for (; ti < seg_end; it += kAGroups) {
                        const int t = resident ? t_begin + ti : t_end - 1 - ti;
                        const int valid = min(128, N - (t - pref[slab]) * 128);
                        if (ok) {
                            ok = role_wait(&ctl->tfull_a[g], uint32_t(it / kAGroups) & 1u, limit, &ctl->abort_flag, a.status);
                            ok = __all_sync(0xffffffffu, ok);
                        }
                        if (ok) {
                            tc_fence_after();
                            // (the last block may hold fewer rows than lanes)
                            if (tk + 1 < a.RA || (g_shifted ? quarter * 32 + 31 >= 128 - rem : quarter * 32 < rem)) {
                                float mk = m[0], lk = l[0];
#pragma unroll
                                for (int k = 1; k < kMaxBlocksA; ++k) if (tk == k) { mk = m[k]; lk = l[k]; }
                                if (valid == 128) lse_fold<false>(lane_addr, valid, scale, mk, lk);
                                else              lse_fold<true>(lane_addr, valid, scale, mk, lk);
#pragma unroll
                                for (int k = 0; k < kMaxBlocksA; ++k) if (tk == k) { m[k] = mk; l[k] = lk; }
                            }
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&ctl->tempty_a[g]);
                        }
                        tk += kAGroups;
                        while (tk >= a.RA) { tk -= a.RA; ++ti; }
                    }
#pragma unroll
                    for (int k = 0; k < kMaxBlocksA; ++k)
                        if (k < a.RA) part[(g * a.RA + k) * 128 + row] = make_float2(m[k], l[k]);
                } else {
                    // this CTA's share of the slab's key sums, which pass B accumulates
                    const int S = min(max(a.n_sent[slab], 0), a.max_sent), P = lc - fc + 1, p = cta - fc;
                    float4* v4 = reinterpret_cast<float4*>(a.vsum + size_t(slab) * a.max_sent * kHeadDim);
                    const int w1 = int((long long)S * 32 * (p + 1) / P);
                    for (int w = int((long long)S * 32 * p / P) + lane; w < w1; w += 32) v4[w] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                named_bar_sync(2, (4 * kAGroups + 1) * 32);
                if (g == 0) {                                // the four groups' parts -> one record per CTA and slab
                    float2* rec = a.rec + size_t(cta + slab) * (size_t(a.RA) * 128);
                    for (int k = 0; k < a.RA; ++k) {
                        float2 x[kAGroups];
                        float M = -INFINITY, L = 0.f;
#pragma unroll
                        for (int q = 0; q < kAGroups; ++q) {
                            const bool sh = k + 1 == a.RA && can_shift && (a.RA == 2 ? q == 3 : (q & 1) != 0);
                            x[q] = part[(q * a.RA + k) * 128 + (sh ? min(row + 128 - rem, 127) : row)];
                            M = fmaxf(M, x[q].x);
                        }
#pragma unroll
                        for (int q = 0; q < kAGroups; ++q) L += x[q].y > 0.f ? x[q].y * ex2f(x[q].x - M) : 0.f;
                        rec[k * 128 + row] = make_float2(M, L);
                    }
                    named_bar_sync(3, 128);
                    if (tid == 64 && ok) { __threadfence(); atomicAdd(a.lse_cnt + slab, uint32_t(hi - lo)); }
                }
                named_bar_sync(4, (4 * kAGroups + 1) * 32);  // the parts have been read
                done = seg_end;
            }
        }
        tc_fence_before();
        named_bar_sync(1, kSweepThreads - 32);               // every accumulator of pass A has been read
        tc_fence_after();
        const int load0 = resident ? 0 : ntl;                // the ring's tiles before pass B
        if (warp < 10 || (warp >= 14 && warp < 18)) {
            // -------------------------------------------------------------- pass B: importance, a thread per token
            const int g = warp < 10 ? (warp - 2) >> 2 : 2;
            const int row = quarter * 32 + lane;
            const uint32_t lane_addr = tmem_base + (uint32_t(quarter * 32) << 16);
            // (what depends on the slab only is kept in registers: while the tensor core streams its operands every look at
            // shared memory takes a hundred cycles and more)
            int slab = slab_of(t_begin), lo = 0, hi = 0, N = 0;         // the slab's tiles are [lo, hi)
            uint32_t ext_no = 0;                             // slabs begun so far
            float *imp_ws = nullptr, *imp_user = nullptr;
            float out_scale = 0.f;                           // 2^-e / window of the slab
            int ti = 0, tk = 0;
            for (int it = 0; it < ntl * a.RB; ++it) {
                const int t = t_begin + ti, i = ti, k = tk;
                if (++tk == a.RB) { tk = 0; ++ti; }
                if (t >= hi) {
                    while (pref[slab + 1] <= t) ++slab;
                    lo = pref[slab]; hi = pref[slab + 1];
                    N = live(slab);
                    out_scale = __uint_as_float(uint32_t(127 - lse_shift(N)) << 23) / float(a.window);
                    imp_ws = a.tok_imp_ws + size_t(slab) * a.max_cap;
                    imp_user = a.tok_imp_user ? a.tok_imp_user + (a.block_table ? size_t(slab) * a.max_pages * 128 : size_t(rowb[slab])) : nullptr;
                    ++ext_no;
                }
                if (it % kBGroups != g) continue;
                if (k == 0 && t == max(lo, t_begin)) {
                    // the group of a slab's first product prepares the slab: log-sum-exp of its query rows from the records of
                    // all its CTAs, negated, in units of raw logits, as three bf16 pieces of the extra K step
                    const int fc = owner(lo), lc = owner(hi - 1);
                    if (lane == 0 && ok) ok = flag_wait(a.lse_cnt + slab, uint32_t(hi - lo), limit, &ctl->abort_flag, a.status);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                    if (ok && ext_no > 1) ok = role_wait(&ctl->extempty, (ext_no - 2) & 1u, limit, &ctl->abort_flag, a.status);
                    ok = __all_sync(0xffffffffu, ok);
                    if (ok) {
                        const float2* r0 = a.rec + size_t(fc + slab) * (size_t(a.RA) * 128);
                        const int n_part = lc - fc + 1;
                        for (int r = row; r < a.R; r += 128) {
                            float M = -INFINITY, L = 0.f;
                            for (int p0 = 0; p0 < n_part; p0 += 8) {         // eight records per round: their loads are in flight together
                                float2 x[8];
#pragma unroll
                                for (int p = 0; p < 8; ++p)
                                    x[p] = p0 + p < n_part ? __ldcg(r0 + size_t(p0 + p) * (a.RA * 128) + r) : make_float2(-INFINITY, 0.f);
                                float mx = M;
#pragma unroll
                                for (int p = 0; p < 8; ++p) mx = fmaxf(mx, x[p].x);
                                L *= M == -INFINITY ? 0.f : ex2f(M - mx);
                                M = mx;
#pragma unroll
                                for (int p = 0; p < 8; ++p) L += x[p].y > 0.f ? x[p].y * ex2f(x[p].x - M) : 0.f;
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
                if (ok) {
                    ok = role_wait(&ctl->tfull_b[g], uint32_t(it / kBGroups) & 1u, limit, &ctl->abort_flag, a.status);
                    ok = __all_sync(0xffffffffu, ok);
                }
                if (!ok) continue;
                tc_fence_after();
                float total = imp_fold<kWB>(lane_addr + g * kBAccCols, n, min(kWB, a.window - k * kWB), scale);
                float* share = tokp + (i & 3) * (a.RB - 1) * 128 + row;
                if (k + 1 < a.RB) {
                    share[k * 128] = total;                  // another group adds the shares up, in the order of the blocks
                } else if (a.RB > 1) {
                    ok = role_wait(&ctl->tokfull[i & 3], uint32_t(i >> 2) & 1u, limit, &ctl->abort_flag, a.status);
                    ok = __all_sync(0xffffffffu, ok);
                    for (int q = a.RB - 2; q >= 0; --q) total += share[q * 128];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (k + 1 < a.RB) mbar_arrive(&ctl->tokfull[i & 3]);
                    mbar_arrive(&ctl->tempty_b[it % (2 * kBGroups)]);
                }
                const int tok = (t - lo) * 128 + row;
                if (k + 1 == a.RB && ok && tok < N) {
                    const float v = total * out_scale;
                    imp_ws[tok] = v;
                    if (imp_user) imp_user[tok] = v;
                }
            }
        } else if (warp < 14) {
            // -------------------------------------------------------------- pass B: per-sentence sums of the key rows
            // The sums are a product on the tensor cores: (tile^T: channel x token) x (indicator: token x sentence slot).
            // A run of consecutive tiles whose sentences all fall among the 16 sentences B .. B + 15 shares one accumulator
            // (slot j = sentence B + j; the products of the run accumulate), so the sums are read out and added to global
            // memory once per run, about every fifth tile.  Each of the four warps writes a quarter of a tile's matrix and
            // arrives; one thread of a fifth warp issues the product; when a tile opens a new run the four warps read out the
            // run before it (a thread owns one channel) while the new one is being multiplied.  A tile that touches more
            // than 16 sentences (empty ones count) gets several matrices, each a run of its own.
            // Every warp keeps, one entry per lane, the sentence offsets B .. B + 31 of the current run (entries past the
            // table read as "never starts"), fetched from global memory when a run opens: loads from shared memory wait
            // several hundred cycles here (the tensor core streams its operands from it), so the per-tile work touches
            // shared memory only to write the matrix.
            constexpr int kNever = 0x7fffffff;
            const int gw = warp - 10;                               // warp of the group: slots 4 gw .. 4 gw + 3 of a matrix
            const int gtid = tid - 320;
            const int ch = quarter * 32 + lane;
            const uint32_t lane_addr = tmem_base + (uint32_t(quarter * 32) << 16) + kPoolCol;
            int slab = slab_of(t_begin), S = 0, N = 0, first = 0;
            int ic = 0;                                             // indicator matrices written so far
            int run = -1, B = 0, w = kNever, w1 = kNever;           // current run: index, sentence of slot 0, offsets B + lane and B + lane + 1
            int wj = kNever, wj1 = kNever;                          // and the offsets of this thread's slot row
            const int sj = 4 * gw + (lane >> 3);                    // the slot row, of which this thread writes two pieces
            int lo = 0, hi = 0, stage = load0 % a.stages;           // the slab's tiles are [lo, hi)
            uint32_t lap = uint32_t(load0 / a.stages);
            uint32_t run_held = 0;                                  // its slots that hold tokens so far
            int run_slab = 0;
            const int32_t* so = a.sent_off;
            // 32-way search for the last sentence that starts at or before token `tok`, one probe per lane
            auto holder = [&](int tok) {
                int lo = 0, len = S;
                while (len > 32) {
                    const int stride = (len + 31) >> 5;
                    const int pidx = lo + lane * stride;
                    const bool le = pidx < lo + len && so[pidx] <= tok;
                    const int adv = max(__popc(__ballot_sync(0xffffffffu, le)) - 1, 0) * stride;
                    len = min(stride, len - adv);
                    lo += adv;
                }
                const bool le = lane < len && so[lo + lane] <= tok;
                return lo + max(__popc(__ballot_sync(0xffffffffu, le)) - 1, 0);
            };
            // read out run r (accumulator r & 1) and add it to the sums
            auto drain = [&](int r, int r_slab, int r_B, uint32_t r_held) {
                ok = role_wait(&ctl->pfull[r & 1], uint32_t(r >> 1) & 1u, limit, &ctl->abort_flag, a.status);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) return;
                tc_fence_after();
                float v[kIndSlots];
                tmem_ld16(lane_addr + uint32_t(r & 1) * kIndSlots, v);
                tc_fence_before();
                float* dst = a.vsum + (size_t(r_slab) * a.max_sent + r_B) * kHeadDim + ch;
#pragma unroll
                for (int j = 0; j < kIndSlots; ++j)
                    if (r_held & (1u << j)) atomicAdd(dst + size_t(j) * kHeadDim, v[j]);
            };
            for (int tl = 0; tl < ntl && ok; ++tl) {
                const int t = t_begin + tl;
                const bool fresh = t >= hi;
                if (fresh) {
                    while (pref[slab + 1] <= t) ++slab;
                    lo = pref[slab]; hi = pref[slab + 1];
                    so = a.sent_off + size_t(slab) * (a.max_sent + 1);
                    S = min(max(a.n_sent[slab], 0), a.max_sent);
                    N = live(slab);
                    // every CTA of the slab has cleared its share of the sums (and left its record)
                    if (lane == 0 && ok) ok = flag_wait(a.lse_cnt + slab, uint32_t(hi - lo), limit, &ctl->abort_flag, a.status);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                    if (!ok) break;
                }
                const int tok0 = (t - lo) * 128, valid = min(128, N - tok0), tok_end = tok0 + valid;
                if (fresh) first = tok0 > 0 ? holder(tok0) : 0;     // (a slab that opens with empty sentences: they get slots)
                // every warp follows every tile's arrival (in order, so it sees each phase of the stage's barrier)
                ok = role_wait(&ctl->full[stage], lap & 1u, limit, &ctl->abort_flag, a.status);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (valid < 128) {
                    // a zero in the indicator does not silence a NaN or an infinity in a dead row: clear the rows past the
                    // slab's end in the staged tile (the logits of those rows are never read)
                    uint8_t* tile = tiles + size_t(stage) * kOpBytes;
                    for (int u = valid * 8 + gtid; u < 128 * 8; u += kPoolWarps * 32) {
                        *reinterpret_cast<uint4*>(tile + u * 16) = make_uint4(0u, 0u, 0u, 0u);
                        *reinterpret_cast<uint4*>(tile + kOpHalfBytes + u * 16) = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
                int cur = first;                                    // first sentence of the tile not yet in a matrix
                int more = 0;
                do {
                    // can the tile (from sentence cur on) join the open run?  its last sentence must be below B + 16
                    bool join = false;
                    if (run >= 0 && !fresh && cur >= B && cur - B < kIndSlots) {
                        const int touching = __popc(__ballot_sync(0xffffffffu, lane > cur - B && B + lane < S && w < tok_end));
                        join = cur + touching - B < kIndSlots;
                    }
                    const int r_prev = run, p_slab = run_slab, p_B = B;
                    const uint32_t p_held = run_held;
                    if (!join) {                                    // open a run at sentence cur
                        ++run; B = cur; run_slab = slab; run_held = 0;
                        w = (B + lane <= S) ? so[B + lane] : kNever;
                        w1 = (B + lane + 1 <= S) ? so[B + lane + 1] : kNever;
                        wj = (B + sj <= S) ? so[B + sj] : kNever;
                        wj1 = (B + sj + 1 <= S) ? so[B + sj + 1] : kNever;
                    }
                    // tile-relative starts of sentences, clamped to the tile; slot j holds the tokens from its start to the next one's
                    auto clamped = [&](int off) { return min(max(min(off, tok_end) - tok0, 0), valid); };
                    const uint32_t held = __ballot_sync(0xffffffffu, lane < kIndSlots && B + lane < S && clamped(w1) > clamped(w));
                    more = __any_sync(0xffffffffu, lane == kIndSlots && B + kIndSlots < S && w < tok_end) ? 1 : 0;    // does slot 15 leave some?
                    const int is = ic & (kIndRing - 1);
                    if (ic >= kIndRing) {                           // the product that read this buffer last has completed
                        ok = role_wait(&ctl->iempty[is], uint32_t(ic / kIndRing - 1) & 1u, limit, &ctl->abort_flag, a.status);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) break;
                    }
                    {
                        const bool is_sent = (held >> sj) & 1u;
                        const int from = is_sent ? clamped(wj) : 0, to = is_sent ? clamped(wj1) : 0;
                        indicator_piece(indb + size_t(is) * kIndBytes, sj, (lane & 7) * 2, from, to);
                        indicator_piece(indb + size_t(is) * kIndBytes, sj, (lane & 7) * 2 + 1, from, to);
                    }
                    fence_proxy_async_smem();                       // the matrix (and cleared rows) are read by the tensor core
                    tc_fence_before();                              // and this warp's reads of the accumulators came first
                    __syncwarp();
                    if (lane == 0) {
                        if (gw == 0) ctl->ind_flags[is] = more | (join ? 2 : 0) | ((!join && r_prev >= 0) ? 4 : 0);
                        mbar_arrive(&ctl->ifull[is]);
                    }
                    run_held |= held;
                    ++ic;
                    if (!join && r_prev >= 0) {                     // the run before, while the new one is being multiplied
                        drain(r_prev, p_slab, p_B, p_held);
                        if (!ok) break;
                    }
                    cur = B + kIndSlots;
                } while (more);
                // the next tile starts in the last sentence of the run's window that starts at or before its first token
                const int n_le = __popc(__ballot_sync(0xffffffffu, B + lane < S && w <= tok0 + 128));
                first = (n_le == 32 && B + 32 < S) ? holder(tok0 + 128) : B + max(n_le - 1, 0);
                if (++stage == a.stages) { stage = 0; ++lap; }
            }
            if (ok && run >= 0) drain(run, run_slab, B, run_held);  // the issuer closes the last run when its tiles are done
        } else {
            // -------------------------------------------------------------- pass B: issuer of the pooling products
            // (its own thread: an issue blocks for the length of the product, and every look at shared memory costs the
            // thread that issues the logits a few hundred cycles)
            {
                const uint32_t leader = elect_leader();
                const uint32_t indb_u32 = smem_u32(indb);
                int pc = 0, run = -1, stage = load0 % a.stages;
                for (int tl = 0; tl < ntl && ok; ++tl) {
                    int flags = 0;
                    do {
                        const int is = pc & (kIndRing - 1);
                        ok = warp_wait(&ctl->ifull[is], uint32_t(pc / kIndRing) & 1u, limit, &ctl->abort_flag, a.status);
                        if (!ok) break;
                        flags = *reinterpret_cast<volatile int*>(&ctl->ind_flags[is]);       // 1: more, 2: joins the run, 4: closes one
                        tc_fence_after();
                        if (flags & 4) umma_commit(&ctl->pfull[run & 1], leader);                    // everything of the run before is issued
                        if (!(flags & 2)) ++run;
                        umma_pool(tmem_base + kPoolCol + uint32_t(run & 1) * kIndSlots, smem_u32(tiles + size_t(stage) * kOpBytes),
                                  indb_u32 + uint32_t(is) * kIndBytes, (flags & 2) != 0, leader);
                        umma_commit(&ctl->iempty[is], leader);
                        ++pc;
                    } while (flags & 1);
                    if (ok) umma_commit(&ctl->empty[stage], leader);
                    if (++stage == a.stages) stage = 0;
                }
                if (ok && run >= 0) umma_commit(&ctl->pfull[run & 1], leader);
                umma_commit(&ctl->retired[2], leader);
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
score_pool_kernel(uint32_t* lse_cnt, int Hk, int max_sent, int max_cap, const int32_t* cap, const int32_t* kv_len,
                  const int32_t* sent_off, const int32_t* n_sent, float eps, const float* tok_imp_ws,
                  const float* vsum, float* sent_imp, __nv_bfloat16* vbar_hi, __nv_bfloat16* vbar_lo, float* sent_lam) {
    pdl_trigger();
    pdl_wait();
    const int slab = blockIdx.y;
    if (blockIdx.x == 0 && threadIdx.x == 0) lse_cnt[slab] = 0u;            // for the next call's sweeps
    const int lane = threadIdx.x & 31;
    const int i0 = blockIdx.x * 8 * kPoolRows + (threadIdx.x >> 5);         // and every eighth after it
    const int S = min(n_sent[slab], max_sent);
    const int N = min(max(kv_len[slab], 0), cap[slab / Hk]);
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
        if (i >= S) break;
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
// Every sentence has four partial sums per block of its slab, each written by one warp: rows by the pair (the four column groups), columns by a
// range's part of J (the four row groups; the blocks of the part's other pairs get zeros).  The CTA that completes a slab adds them up in
// order, so the results do not depend on who was first.  They lie where the sums of the keys were, which the pooling was the last to read.
// The penalty is the maximum over later sentences; only those beyond tau are reported, which are few (pass 1, an integer maximum).
// Roles as in the token-level kernel: a TMA warp, two MMA warps that take the pairs in turn, sixteen epilogue warps with 32
// rows x 32 columns of every accumulator each, column sums in registers for as long as J stays.
// Three shared-memory slots hold a block's high and low parts.  One is J's, the other two take the I blocks in turn; the next J takes
// the slot that is free next and the old J's goes to the end of the queue, so a change of J costs no drain.
// Bound by its epilogue: 2.4 and 2.1 us a pair (passes 1 and 2, about 130 pairs per SM) against 0.8 us for the three products, which stream
// 192 KB of operands at the shared-memory port's 128 bytes per clock.  The four warps of a scheduler are in the same phase of the
// same pair, and column sums leave no registers for two pairs at once.  Half the products and half the exponentials of evaluating
// all pairs twice: 128 slabs x 2K sentences, the whole scoring call: 2319 -> 2190 us.
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
    alignas(16) float colz[16][32];          // pass 2, by epilogue warp: 1 / Z_j of its columns
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
    int slab, S, J, t;                       // pair t of block column J: 0 is the diagonal, t > 0 multiplies block t - 1
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
    __device__ __forceinline__ bool next(const int* ipref) {
        --left;
        if (t++ < J) return false;
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
    const int first = int(total * blockIdx.x / gridDim.x), count = int(total * (blockIdx.x + 1) / gridDim.x) - first;

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
                    const int row = w.slab * max_sent + block * 128;
                    mbar_expect_tx(&ctl->full[s][part], kOpBytes);
                    tma_load_2d(dst, map, 0, row, &ctl->full[s][part]);
                    tma_load_2d(dst + kOpHalfBytes, map, 64, row, &ctl->full[s][part]);
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
        const int quarter = warp & 3, c0 = ((warp - 4) >> 2) * 32;   // this warp's rows (32 * quarter + lane) and columns
        const uint32_t lane_addr = tmem_base + (uint32_t(quarter * 32) << 16) + c0;
        float* colz_s = ctl->colz[warp - 4];
        const float2* colz = reinterpret_cast<const float2*>(colz_s);
        float2 cs[16];
        bool ok = true, fresh = true;
        uint32_t acc = 0, parity = 0;
        int done = 0;                                                // pairs of this slab in this range
        int cslot = 0;                                               // whose partial the column sums become
        uint32_t* lam_bits = reinterpret_cast<uint32_t*>(sent_lam);
        GramWalk w;
        w.start(ipref, first, count);
        w.S = count > 0 ? sent_of(w.slab) : 0;
#pragma unroll 1
        while (w.left > 0) {
            const size_t base = size_t(w.slab) * max_sent;
            const int j0 = w.J * 128 + c0;
            const bool diag = w.t == 0;
            const int ib = diag ? w.J : w.t - 1, i = ib * 128 + quarter * 32 + lane;
            float* p_slab = parts + size_t(w.slab) * parts_slab;         // [4 * blocks][max_sent]
            if (fresh) {
#pragma unroll
                for (int k = 0; k < 16; ++k) cs[k] = make_float2(0.f, 0.f);
                cslot = ib;
                if (kPass == 2) {
                    const float z = j0 + lane < w.S ? sc_z[base + j0 + lane] : 0.f;
                    __syncwarp();
                    colz_s[lane] = z > 0.f ? 1.f / z : 0.f;
                    __syncwarp();
                }
            } else if (j0 + lane < w.S) {
                p_slab[size_t(ib * 4 + quarter) * max_sent + j0 + lane] = 0.f;
            }
            float invz_i = 0.f;                                      // pass 2: 1 / Z_i, the weight of this row in column sums
            if (kPass == 2 && i < w.S) { const float z = sc_z[base + i]; invz_i = z > 0.f ? 1.f / z : 0.f; }
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
                float2 row = make_float2(0.f, 0.f);
                const float2 l2 = make_float2(kLog2e, kLog2e), iz2 = make_float2(invz_i, invz_i);
                auto add = [&](int k, float2 e) {
                    if (kPass == 1) {
                        row = __fadd2_rn(row, e);
                        cs[k] = __fadd2_rn(cs[k], e);
                    } else {
                        row = __ffma2_rn(e, colz[k], row);
                        cs[k] = __ffma2_rn(e, iz2, cs[k]);
                    }
                };
                float mx = -INFINITY;
                if (!diag && (w.J + 1) * 128 <= w.S) {               // (I < J: all rows are the slab's)
                    if (kPass == 1) {
                        float m1 = -INFINITY;
#pragma unroll
                        for (int k = 0; k < 32; k += 4) { mx = max3(mx, v[k], v[k + 1]); m1 = max3(m1, v[k + 2], v[k + 3]); }
                        mx = fmaxf(mx, m1);
                    }
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const float2 x = __fmul2_rn(make_float2(v[2 * k], v[2 * k + 1]), l2);
                        add(k, make_float2(ex2f(x.x), ex2f(x.y)));
                    }
                } else {                                             // nothing where a row or column is none of the slab's, and for i == j
                    const int lim = i < w.S ? w.S - j0 : 0, self = i - j0;
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const bool x = 2 * k < lim, y = 2 * k + 1 < lim;
                        if (kPass == 1) {
                            if (x && 2 * k > self) mx = fmaxf(mx, v[2 * k]);
                            if (y && 2 * k + 1 > self) mx = fmaxf(mx, v[2 * k + 1]);
                        }
                        add(k, make_float2(x && 2 * k != self ? ex2f(v[2 * k] * kLog2e) : 0.f,
                                           y && 2 * k + 1 != self ? ex2f(v[2 * k + 1] * kLog2e) : 0.f));
                    }
                }
                if (kPass == 1 && mx > tau && !ext.table) atomicMax(lam_bits + base + i, ordered_bits(mx));
                // (the diagonal pair is symmetric: its column sums are all there is to it)
                if (!diag && i < w.S) p_slab[size_t(w.J * 4 + (c0 >> 5)) * max_sent + i] = row.x + row.y;
            }
            if (++acc == kGramAcc) { acc = 0; parity ^= 1u; }
            ++done;
            const int slab = w.slab, S = w.S;
            fresh = w.next(ipref);
            if ((fresh || w.left == 0) && ok) {
                float s[32];
#pragma unroll
                for (int k = 0; k < 16; ++k) { s[2 * k] = cs[k].x; s[2 * k + 1] = cs[k].y; }
                const float sum = col_reduce32(s, lane);
                if (j0 + lane < S) p_slab[size_t(cslot * 4 + quarter) * max_sent + j0 + lane] = sum;
            }
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
                        float sum = 0.f;
#pragma unroll 4
                        for (int q = 0; q < nb; ++q) {
                            const float* p = p_slab + size_t(q * 4) * max_sent + k;
                            sum += (__ldcg(p) + __ldcg(p + max_sent)) + (__ldcg(p + 2 * size_t(max_sent)) + __ldcg(p + 3 * size_t(max_sent)));
                        }
                        const size_t o = base + k;
                        if (kPass == 1) {
                            sc_z[o] = sum;
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
                done = 0;
                w.S = w.left > 0 ? sent_of(w.slab) : 0;
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
constexpr int kSmallSent = 128;
constexpr int kSmallBatch = 8;          // sentences of a warp: their loads are in flight together
struct SmallCtl {
    uint64_t done;
    uint32_t tmem_base;
    alignas(16) float imp[kSmallSent], sum[4][kSmallSent], mx[4][kSmallSent], red[4][kSmallSent], invz[kSmallSent];
};
constexpr size_t kSmallSmem = 1024 + 2 * size_t(kOpBytes) + sizeof(SmallCtl);

__global__ void __launch_bounds__(kSmallThreads)
score_small_kernel(uint32_t* lse_cnt, int Hk, int max_sent, int max_cap, const int32_t* cap, const int32_t* kv_len, const int32_t* sent_off,
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
    if (tid == 0) lse_cnt[slab] = 0u;                    // for the next call's sweeps
    const int S = min(max(n_sent[slab], 0), max_sent), N = min(max(kv_len[slab], 0), cap[slab / Hk]);
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

    CUtensorMap mapK, mapQ, mapHi, mapLo;
    if (int rc = tmap_rows(&mapK, K, uint64_t(shape->total_rows), 128)) return rc;
    if (int rc = tmap_qwin(&mapQ, q_win, uint64_t(shape->batch) * Hq, uint32_t(shape->window), uint32_t(L.sc_wb), uint32_t(n)))
        return rc;
    const uint64_t vrows = uint64_t(L.slabs) * uint64_t(shape->max_sent);
    if (int rc = tmap_rows(&mapHi, vbar_hi, vrows, 128)) return rc;
    if (int rc = tmap_rows(&mapLo, vbar_lo, vrows, 128)) return rc;

    SweepArgs a{};
    a.Hq = Hq; a.Hk = Hk; a.window = shape->window; a.n_slabs = L.slabs; a.max_cap = shape->max_cap;
    a.max_sent = shape->max_sent;
    a.WB = L.sc_wb; a.RB = L.sc_rb; a.N = L.sc_wb * n; a.R = a.RB * a.N; a.RA = L.sc_ra;
    a.slab_off = shape->slab_off; a.cap = shape->cap; a.kv_len = kv_len; a.sent_off = sent_off; a.n_sent = n_sent;
    a.rec = reinterpret_cast<float2*>(w + L.sc_part); a.lse_cnt = reinterpret_cast<uint32_t*>(w + L.sc_cnt);
    a.tok_imp_user = tok_imp; a.tok_imp_ws = sc_tok; a.vsum = vsum; a.status = status;
    a.hdr = reinterpret_cast<const Header*>(w + L.header);
    a.block_table = block_table; a.max_pages = max_pages;
    const size_t max_smem = 227 * 1024;
    size_t fixed = 1024 + size_t(a.R) * kRowBytes + size_t(kIndRing) * kIndBytes + 128 * kExtRow + size_t(a.RA) * 128 * kExtRow +
                   sizeof(SweepCtl) + size_t(a.RB - 1) * 4 * 128 * 4;
    // The table of slabs (8 bytes each) goes into shared memory as long as one tile stage fits beside it: all but windows of some hundred
    // query rows with a thousand slabs and more.  A 512-row window leaves room for 900 slabs; without the other form the call would end there.
    const size_t table_bytes = size_t(2 * L.slabs + 1) * 4;
    const bool in_global = fixed + table_bytes + kOpBytes > max_smem;
    if (in_global) a.table = reinterpret_cast<int*>(w + L.slab_table);
    else fixed += table_bytes;
    const size_t gsmem = gram_smem_bytes(L.slabs);
    if (shape->max_sent > kSmallSent && gsmem > max_smem) {          // (before anything is enqueued)
        set_error_text("skipkv_score: more than 128 sentences per slab and batch * n_kv_heads too large for the shared-memory table of the Gram kernels");
        return SKIPKV_ERR_UNSUPPORTED;
    }
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
    // one tile of sentences per slab: one kernel instead of three, with the operands in shared memory throughout
    if (shape->max_sent <= kSmallSent) {
        SKIPKV_CUDA(launch_dependent(score_small_kernel, dim3(L.slabs), dim3(kSmallThreads), kSmallSmem, st, a.lse_cnt, Hk, int(shape->max_sent),
                                     int(shape->max_cap), shape->cap, kv_len, sent_off, n_sent, params->eps, params->sigma,
                                     params->tau, static_cast<const float*>(sc_tok), static_cast<const float*>(vsum), sent_imp,
                                     sent_red, sent_lam, sent_score, ext, reinterpret_cast<const Header*>(w + L.header)));
        return SKIPKV_OK;
    }
    {
        dim3 pgrid((shape->max_sent + 8 * kPoolRows - 1) / (8 * kPoolRows), L.slabs);
        SKIPKV_CUDA(launch_dependent(score_pool_kernel, pgrid, dim3(256), 0, st, a.lse_cnt, Hk, shape->max_sent, shape->max_cap,
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
