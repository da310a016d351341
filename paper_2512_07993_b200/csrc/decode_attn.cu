// skipkv_decode_attn: GQA decode attention over the ragged, compacted cache (the attention
// equation of paper Section 4.1 with one query per head), with the steering add of Section 4.2
// performed by the same launch.
//
// The step is HBM bound: every live K and V row is read exactly once, 512 bytes per token and slab, and what a call
// costs beyond that is latency: a decode step is a chain of launches (one per layer) over caches of a few thousand rows.
// Design:
//  * Work = 64-row tiles enumerated over all (sequence, head) slabs.  The tile list is cut into equal contiguous
//    ranges, one per CTA (one CTA per SM), so CTAs are balanced whatever the ragged lengths are; a CTA's range may
//    cross slab boundaries, each (CTA, slab) intersection gives one partial result (max, sum, 128 accumulators per head).
//  * Four warps, each with its own 16 rows of every tile and its own ring of asynchronous 16-byte copies: no barrier and
//    no mbarrier in the stream.  Copies (not bulk copies) because the rows are written to shared memory with their
//    16-byte pieces permuted (piece c of row r at c ^ (r & 7)), which makes the matrix loads free of bank conflicts, and
//    because rows past the slab's end are zero-filled and the row being appended can come from another pointer.
//    Three stages of 8 KB per warp keep 64 KB in flight per SM while 32 KB are worked on.
//  * Math on the tensor cores (mma.sync m16n8k16: one query row per head is far below a tcgen05 tile): S^T = K Q^T with 16
//    tokens as rows and the group's heads as the eight columns, then (P V)^T = V^T P^T with 16 channels as rows.  The probabilities
//    go in as three bf16 parts (transposed in registers by movmatrix), which together are the fp32 value, and the products of a
//    tile are added to the sums over the tiles in fp32 with rounding: the tensor core's own accumulation truncates.  With two
//    parts and sums kept in the tensor core 1 to 3 outputs in a thousand were not the exact result rounded to bf16; now 0.2 to 0.5,
//    as with fp32 arithmetic throughout.  Any group size costs the same up to four heads, and the same from five to eight.
//    There is one warp to a scheduler, so a tile is a chain of latencies (16 x 8 x 16 products 10 clocks apart and 30 long, exchanges
//    24, matrix loads 16): independent chains of products, exchanges of the heads' maxima only when one of them rises.
//    Against the two parts: 72.8 -> 74.4 us (two steps of 80 slabs x 4.1K rows), 163.2 -> 168.6 (80 slabs of 16K to 32K), 96.8 -> 104.5
//    (128 slabs x 8.2K, five heads).
//  * Little shared memory and few threads, so that the CTAs of the next launch are resident while this one streams: a
//    programmatic dependent launch derives its tile schedule and starts its first tiles towards L2 before the launch
//    ahead of it has finished, and only then waits.  Behind the wait the first copies go out under that schedule at once; what was read
//    early is checked while they are on their way (see "schedule").  With the check, the steering operands and the queries one round trip
//    after the other in front of the first tile a step of one sequence x 2048 rows took 9.97 us a layer, with them together 8.9.
//  * Straight-line code counts: a launch behind other kernels (the products of a model's layer) finds its code in no instruction cache, and
//    all that stands before the first copies is fetched first, about eight instructions a line.  So what runs once or seldom is rolled up, and the
//    first copies are one piece of code for both attempts.  With the loops unrolled as the compiler saw fit and two pieces, behind four matrix
//    products: 80 slabs x 4.1K rows 48.4 -> 45.2 us, two sequences of 8K 34.3 -> 30.0, 80 slabs of 16K to 32K 166 -> 163, 128 slabs x 8.2K
//    (five heads) 108 -> 103; a step of one sequence x 2048 rows, 32 launches back to back, 281.6 -> 271.
//  * Softmax is online in base 2 with a warp-uniform lazy rescale.
//  * The last CTA to deliver a partial for a slab (self-resetting counter in the workspace) merges that slab's partials.
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "steer.cuh"

namespace skipkv {

constexpr int kDecWarps = 4;
constexpr int kDecThreads = kDecWarps * 32;
constexpr int kWarpRows = 16;                             // rows of a tile that one warp works on
constexpr int kTileRows = kDecWarps * kWarpRows;          // 64
constexpr int kPageRows = 128;                            // paged cache: rows per page
constexpr int kStages = 3;
constexpr int kStageBytes = 2 * kWarpRows * kRowBytes;    // one warp's K rows, then its V rows
constexpr int kRingBytes = kDecWarps * kStages * kStageBytes;
constexpr int kPrefetchTiles = 3;                         // tiles a CTA starts towards L2 before it may read the cache
constexpr int kTriggerTiles = 2;                          // tiles a CTA still has when it lets the next launch's CTAs start
constexpr int kPartStride = kDecPartStride;               // record of one head: 128 accumulators, max, sum (16-byte aligned rows)
constexpr int kWpStride = 132;                            // the same in shared memory
constexpr int kMaxDecSlabs = 8192;
constexpr int kDecMaxGrid = 256;

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 16 bytes global -> shared, asynchronously; src_bytes = 0 writes zeros and reads nothing
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// D[16 x 8] += A[16 x 16] B[16 x 8], bf16 operands, fp32 accumulators
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the same without a sum to add to
__device__ __forceinline__ void mma16816_first(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// Two probabilities as three bf16 parts each, the leading, middle and last 8 bits of the fp32 values.
__device__ __forceinline__ uint32_t top_halves(float2 x) { return __byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x7632); }
__device__ __forceinline__ float2 without_top(float2 x) {
    const float2 top = make_float2(__uint_as_float(__float_as_uint(x.x) & 0xffff0000u), __uint_as_float(__float_as_uint(x.y) & 0xffff0000u));
    return __ffma2_rn(top, make_float2(-1.f, -1.f), x);
}
__device__ __forceinline__ void split_bf16(float2 x, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    hi = top_halves(x);
    x = without_top(x);
    mid = top_halves(x);
    lo = top_halves(without_top(x));
}
// Adds 1; the CTA's stores before its last barrier come first, and what the CTAs that arrived earlier stored is visible behind the next one.
__device__ __forceinline__ uint32_t arrive_acq_rel(uint32_t* p) {
    uint32_t old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
    return old;
}
// an 8 x 8 matrix of bf16 pairs across the warp, transposed
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

// Optional fusion of the per-step bookkeeping into the decode launch (k_new == nullptr: plain decode attention).
// The tile schedule covers the cached rows and the new one, which is read from k_new / v_new; the CTA that owns a slab's
// last tile also writes the new row into the cache and updates the slab's range list and length.  Lengths are read from
// kv_len and written to kv_len_out (a different buffer), so CTAs that start late still derive the same tile schedule.
struct StepArgs {
    const uint4* k_new;          // [batch][Hk][16]
    const uint4* v_new;
    int32_t* kv_len_out;         // [batch][Hk]
    int32_t* sent_off;           // range list, updated in place
    int32_t* sent_id;
    int32_t* n_sent;
    const uint8_t* new_sent;     // [batch]
    const int32_t* gen_id;       // [batch]
    uint4* q_win;                // nullable: [batch][Hq][window][16]
    int window, slot, max_sent;
};

// kStep: the launch also performs the per-step bookkeeping described at StepArgs (a separate instance, so that
// plain decode attention carries none of it).
// kFew: up to four heads per group.  The eight columns of an operand are then the heads twice: the high parts of the probabilities
// in the first four, the middle ones in the others, so that two products do the work of three.
template <bool kStep, bool kFew>
__global__ void __launch_bounds__(kDecThreads, 2)
decode_attn_kernel(int batch, int Hq, int Hk, int n_slabs, long long total_rows, const int64_t* slab_off, const int32_t* cap,
                   const __nv_bfloat16* q, const uint8_t* K, const uint8_t* V, const int32_t* kv_len,
                   __nv_bfloat16* out, uint32_t* status, uint32_t* dec_cnt, float* dec_part, int d_model,
                   __nv_bfloat16* hidden, const __nv_bfloat16* steer_vec, const float* alpha, const uint8_t* flag,
                   const int32_t* block_table, int max_pages, StepArgs step) {
    extern __shared__ __align__(128) uint8_t dsm[];
    const int n = Hq / Hk;                                                   // heads per group
    float* wpart = reinterpret_cast<float*>(dsm + kRingBytes);               // [warps][n heads][132]
    int* pref = reinterpret_cast<int*>(wpart + kDecWarps * n * kWpStride);   // [n_slabs + 1] tile prefix
    uint32_t* lens = reinterpret_cast<uint32_t*>(pref + n_slabs + 1);        // [n_slabs] 2 * rows to attend to + (a row is appended)
    __shared__ uint32_t s_wsum[kDecWarps];
    __shared__ int s_last;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, cta = blockIdx.x;
    // rows slab s has room for; with a block table (paged cache) no more than its max_pages pages
    auto room = [&](int s) { return block_table ? min(cap[s / Hk], max_pages * kPageRows) : cap[s / Hk]; };
    auto slab_len = [&](int s) {
        const int r = room(s), old = min(max(kv_len[s], 0), r);
        const uint32_t app = kStep && old < r ? 1u : 0u;
        return (uint32_t(old) + app) * 2u + app;
    };
    // cache row of token t of slab s (contiguous slabs, or through the block table)
    auto phys_row = [&](int s, int t) {
        return block_table ? size_t(max(block_table[size_t(s) * max_pages + t / kPageRows], 0)) * kPageRows + size_t(t % kPageRows)
                           : slab_row0(slab_off, cap, Hk, s / Hk, s % Hk) + size_t(t);
    };

    // ---- schedule.  The lengths may be written by the launch ahead of this one, but mostly they are older (another layer
    // ran in between).  So the tile schedule is derived from what they are now, the first tiles of this CTA are started
    // towards L2 (the point of coherence, so a row that is still being written is not read too early), and after the wait
    // the lengths are read once more: only if one of them changed is the schedule derived again.
    const int s_per = (n_slabs + kDecThreads - 1) / kDecThreads;
    const int s_lo = min(tid * s_per, n_slabs), s_hi = min(s_lo + s_per, n_slabs);
#pragma unroll 1
    for (int s = s_lo; s < s_hi; ++s) lens[s] = slab_len(s);
    auto tiles_of = [&](int s) { return (int(lens[s] >> 1) + kTileRows - 1) / kTileRows; };
    cta_prefix<kDecThreads>(n_slabs, tiles_of, pref, s_wsum);
    // CTA c has the tiles [c T / Ge, (c + 1) T / Ge) of the T tiles, Ge = the CTAs that have work
    int T, Ge, t_begin, t_end, slab0;
    auto derive = [&]() {
        T = pref[n_slabs];
        Ge = min(G, T);
        t_begin = cta < Ge ? int((long long)cta * T / Ge) : T;
        t_end = cta < Ge ? int((long long)(cta + 1) * T / Ge) : T;
        int lo = 0, hi = n_slabs - 1;                     // slab holding tile t_begin: the last s with pref[s] <= t_begin
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pref[mid] <= t_begin) lo = mid; else hi = mid - 1;
        }
        slab0 = lo;
    };
    derive();
    if (tid < 2 * kPrefetchTiles && t_begin + (tid >> 1) < t_end) {
        const int t = t_begin + (tid >> 1);
        int s = slab0;
        while (pref[s + 1] <= t) ++s;
        const int r0 = (t - pref[s]) * kTileRows;
        const int rows = min(kTileRows, int(lens[s] >> 1) - int(lens[s] & 1u) - r0);     // without the row not yet written
        const long long row = (long long)phys_row(s, r0);
        if (rows > 0 && row >= 0 && row + rows <= total_rows)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(((tid & 1) ? V : K) + size_t(row) * kRowBytes),
                         "r"(rows * kRowBytes) : "memory");
    }
    if (kStep) {                                          // the rows being appended are read in the middle of the stream
        const size_t bytes = size_t(n_slabs) * kRowBytes;
#pragma unroll 1
        for (size_t o = size_t(cta * kDecThreads + tid) * 128; o < bytes; o += size_t(G) * kDecThreads * 128) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(step.k_new) + o));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(step.v_new) + o));
        }
    }
    // Row of token 0 of the first slab (paged: the page of the CTA's first tile).  What is read here before the wait is used after it, for the
    // first copies, and checked like the lengths while they are on their way; rows outside the buffers make it count as changed at once.
    auto first_row = [&]() {
        if (t_begin >= t_end) return size_t(0);
        const int r = (t_begin - pref[slab0]) * kTileRows;
        return block_table ? size_t(max(block_table[size_t(slab0) * max_pages + r / kPageRows], 0)) : slab_row0(slab_off, cap, Hk, slab0 / Hk, slab0 % Hk);
    };
    size_t row_first = first_row();
    const bool early = t_begin < t_end &&
        (long long)(block_table ? (row_first + 1) * kPageRows : row_first + (lens[slab0] >> 1)) <= total_rows && (long long)row_first >= 0;
    pdl_wait();                                           // inputs (and the workspace) may come from the kernel before

    // ---- copies: this warp's 16 rows of the CTA's k-th tile go to stage k % kStages.  The cursor walks the slab parts of
    // the tile range; divisions and table reads happen once per part.  unchecked: under the schedule from before the wait.
    const uint32_t ring = smem_u32(dsm) + warp * kStages * kStageBytes;
    const int c_col = lane & 15, c_half = lane >> 4;
    int p_t = t_begin, p_slab = slab0, p_end = t_begin, p_r0 = 0, p_rows = 0, p_stage = 0;
    size_t p_row0 = 0;
    bool p_app = false;
    long long bound = total_rows;                         // of the unchecked copies, until the schedule is confirmed
    long long far = 0;                                    // where the farthest of the unchecked copies ends
    auto issue_next = [&](auto unchecked) {
        if (p_t < t_end) {
            if (p_end <= p_t) {
                while (pref[p_slab + 1] <= p_t) ++p_slab;
                p_end = pref[p_slab + 1];
                p_r0 = (p_t - pref[p_slab]) * kTileRows + warp * kWarpRows;
                p_rows = int(lens[p_slab] >> 1);
                p_app = kStep && (lens[p_slab] & 1u);
                if (!block_table) p_row0 = p_t == t_begin ? row_first : slab_row0(slab_off, cap, Hk, p_slab / Hk, p_slab % Hk);
            }
            const int rows = p_rows - p_r0;               // rows of this warp's part, may be <= 0 or > 16
            if (rows > 0) {
                size_t row = p_row0 + size_t(p_r0);
                if (block_table)
                    row = (p_t == t_begin ? row_first : size_t(max(block_table[size_t(p_slab) * max_pages + p_r0 / kPageRows], 0))) * kPageRows +
                          size_t(p_r0 % kPageRows);
                // (never beyond the buffers, also under lengths that turn out to be old; from one that is left out on all are, and count as changed)
                if (decltype(unchecked)::value) far = max(far, (long long)row + min(rows, kWarpRows));
                if (!decltype(unchecked)::value || far <= bound) {
                    const size_t off = (row + size_t(c_half)) * kRowBytes + size_t(c_col) * 16;
                    const uint8_t *kp = K + off, *vp = V + off;
                    // (row 2 i + c_half takes its pieces at c_col ^ ((2 i + c_half) & 7): four addresses and constant distances from them)
                    const uint32_t dst = ring + p_stage * kStageBytes + c_half * kRowBytes + ((c_col ^ c_half) << 4);
                    const int last = rows - 1;                // the appended row, where there is one
                    if (rows > kWarpRows || (rows == kWarpRows && !p_app)) {
#pragma unroll
                        for (int i = 0; i < kWarpRows / 2; ++i) {
                            const uint32_t d = (dst ^ ((i & 3) << 5)) + i * 2 * kRowBytes;
                            cp_async16(d, kp + i * 2 * kRowBytes);
                            cp_async16(d + kWarpRows * kRowBytes, vp + i * 2 * kRowBytes);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < kWarpRows / 2; ++i) {
                            const int r = 2 * i + c_half;
                            const uint32_t d = (dst ^ ((i & 3) << 5)) + i * 2 * kRowBytes;
                            const void *ks = kp + i * 2 * kRowBytes, *vs = vp + i * 2 * kRowBytes;
                            if (kStep && p_app && r == last) {
                                ks = step.k_new + size_t(p_slab) * 16 + c_col;
                                vs = step.v_new + size_t(p_slab) * 16 + c_col;
                            }
                            const int bytes = r <= last ? 16 : 0;
                            cp_async16(d, bytes ? ks : K, bytes);
                            cp_async16(d + kWarpRows * kRowBytes, bytes ? vs : V, bytes);
                        }
                    }
                }
            }
            p_r0 += kTileRows;
            ++p_t;
            if (++p_stage == kStages) p_stage = 0;
        }
        cp_async_commit();                                // empty groups keep the count
    };
    // Everything that comes from memory before the first tile is requested at once, in the order in which it is needed, and consumed behind the
    // first copies: the lengths and the first row once more; the first slab's queries; the operands of the steering add and (fused
    // step) this step's queries for their slot of the observation window, both independent of the attention (consecutive warps' shares
    // lie in different CTAs).
    const uint32_t len_again = s_lo < s_hi ? slab_len(s_lo) : 0u;
    const size_t row_again = first_row();
    const int g = lane >> 2, qd = lane & 3;               // mma fragments: rows (tokens, channels) g and g + 8, columns (heads) 2 qd and 2 qd + 1
    uint32_t qa[8][2];
    auto load_q = [&](int slab_) {
        const int hd = kFew ? g & 3 : g;                  // head of this lane's column
        const uint32_t* qp = reinterpret_cast<const uint32_t*>(q + (size_t(slab_ / Hk) * Hq + size_t(slab_ % Hk) * n + min(hd, n - 1)) * kHeadDim) + qd;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            qa[ks][0] = hd < n ? qp[ks * 8] : 0u;
            qa[ks][1] = hd < n ? qp[ks * 8 + 4] : 0u;
        }
    };
    int q_slab = slab0;
    if (t_begin < t_end) load_q(slab0);
    const int side0 = (warp * G + cta) * 32 + lane, side_step = G * kDecThreads;
    const int vec_per_row = d_model / 8, steer_total = hidden != nullptr ? batch * vec_per_row : 0;
    const int qwin_total = kStep && step.q_win != nullptr ? batch * Hq * 16 : 0;
    SteerVec st = {};
    uint4 qw = make_uint4(0u, 0u, 0u, 0u);
    if (side0 < steer_total) st = steer_load(side0, vec_per_row, hidden, steer_vec, alpha, flag);
    if (side0 < qwin_total) qw = reinterpret_cast<const uint4*>(q)[side0];
    bool go = early;
#pragma unroll 1
    for (int attempt = 0;; ++attempt) {
        if (go) {
#pragma unroll 1
            for (int k = 0; k < kStages - 1; ++k) issue_next(std::true_type{});
        }
        if (attempt > 0) break;
        int changed = row_again != row_first || far > total_rows;
        if (s_lo < s_hi && len_again != lens[s_lo]) changed = 1;
#pragma unroll 1
        for (int s = s_lo + 1; s < s_hi; ++s)
            if (slab_len(s) != lens[s]) changed = 1;
        changed = __syncthreads_or(changed);              // (no thread writes a length before all have compared theirs)
        if (early && !changed) break;
        if (changed) {
            cp_async_wait<0>();
#pragma unroll 1
            for (int s = s_lo; s < s_hi; ++s) lens[s] = slab_len(s);
            cta_prefix<kDecThreads>(n_slabs, tiles_of, pref, s_wsum);
            derive();
            row_first = first_row();
            p_t = p_end = t_begin; p_slab = slab0; p_stage = 0;
            q_slab = -1;
        }
        bound = 0x7fffffffffffffffll;
        go = true;
    }
    // The next launch's CTAs may start when every CTA has come here: early enough to have their schedule and their first
    // tiles ready, and not so early that what they start towards L2 is evicted by this launch's stream.
    bool triggered = false;
    auto maybe_trigger = [&](int tiles_left) {
        if (!triggered && tiles_left <= kTriggerTiles) { triggered = true; pdl_trigger(); }
    };
    maybe_trigger(t_end - t_begin);
    auto qwin_at = [&](int i) { return step.q_win + (size_t(i >> 4) * step.window + step.slot) * 16 + (i & 15); };
    if (side0 < steer_total) steer_store(side0, vec_per_row, hidden, st);
    if (side0 < qwin_total) *qwin_at(side0) = qw;
#pragma unroll 1
    for (int i = side0 + side_step; i < steer_total; i += side_step)
        steer_store(i, vec_per_row, hidden, steer_load(i, vec_per_row, hidden, steer_vec, alpha, flag));
#pragma unroll 1
    for (int i = side0 + side_step; i < qwin_total; i += side_step) *qwin_at(i) = reinterpret_cast<const uint4*>(q)[i];
    // fused step: new length and range list of a slab after the append (every thread has read n_sent before any calls this)
    auto step_tables = [&](int slab_, int b_, int new_len, bool appended, int S0, int starts_sentence) {
        int32_t* so = step.sent_off + size_t(slab_) * (step.max_sent + 1);
        const bool table_ok = S0 >= 0 && S0 <= step.max_sent;
        int S = S0;
        bool full_list = false;
        if (appended && table_ok && (S0 == 0 || starts_sentence)) {
            if (S0 < step.max_sent) S = S0 + 1; else full_list = true;   // full list: the token joins the last sentence
        }
        if (tid == 0) {
            step.kv_len_out[slab_] = new_len;
            if (appended && table_ok && S != S0) {
                if (S0 == 0) so[0] = 0;
                step.sent_id[size_t(slab_) * step.max_sent + S0] = step.gen_id[b_];
                step.n_sent[slab_] = S;
            }
            if (!appended || !table_ok || full_list) atomicOr(status, SKIPKV_STATUS_BAD_TABLE);
        }
        if (appended && table_ok)
#pragma unroll 1
            for (int i = S + tid; i <= step.max_sent; i += kDecThreads) so[i] = new_len;
    };

    const float qscale = 1.4426950408889634f * rsqrtf(float(kHeadDim));
    const float2 qscale2 = make_float2(qscale, qscale);
    // this lane's row address offsets inside a stage for the matrix loads (K: token octets by the upper bit, V: by the lower)
    const int lm = lane >> 3, k_row = (lane & 7) + (lm >> 1) * 8, v_row = (lane & 7) + (lm & 1) * 8;
    // piece 2 ks + x of a row lies at (2 ks + x) ^ (row & 7): the addresses of steps 0 to 3 differ in two bits, steps 4 to 7 are 128 bytes on
    const uint32_t k_base = ring + k_row * kRowBytes + (((lm & 1) ^ (lane & 7)) << 4);
    const uint32_t v_base = ring + (kWarpRows + v_row) * kRowBytes + (((lm >> 1) ^ (lane & 7)) << 4);

    int slab = slab0, t = t_begin, c_stage = 0;
    while (t < t_end) {
        // -------------------------------------------------------------- one (CTA, slab) segment
        while (pref[slab + 1] <= t) ++slab;
        const int seg_end = min(t_end, pref[slab + 1]);
        const int b = slab / Hk, h = slab % Hk;
        const int n_rows = int(lens[slab] >> 1);
        const bool appended = kStep && (lens[slab] & 1u);
        const bool own_tail = kStep && seg_end == pref[slab + 1];
        int step_S0 = 0, step_starts = 0;
        uint4 new_piece = make_uint4(0u, 0u, 0u, 0u);
        size_t new_at = 0;
        if (own_tail) {
            step_S0 = step.n_sent[slab]; step_starts = step.new_sent[b];
            if (appended && warp == kDecWarps - 1) {      // the row being appended, which goes into the cache behind the tiles
                new_piece = (c_half ? step.v_new : step.k_new)[size_t(slab) * 16 + c_col];
                new_at = phys_row(slab, n_rows - 1) * 16 + c_col;
            }
        }
        if (slab != q_slab) { load_q(slab); q_slab = slab; }
        float2 acc[8][2];                                 // channels 16 j + g and 16 j + 8 + g of the lane's two heads
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
        float2 m = make_float2(-INFINITY, -INFINITY), l = make_float2(0.f, 0.f);    // their running maximum, this lane's share of the sum
        int rows_left = n_rows - (t - pref[slab]) * kTileRows - warp * kWarpRows;     // of this warp's part of the tile
        for (; t < seg_end; ++t, rows_left -= kTileRows) {
            cp_async_wait<kStages - 2>();
            __syncwarp();                                 // every lane's pieces have landed; the stage before is read out
            issue_next(std::false_type{});
            maybe_trigger(t_end - t);
            if (rows_left > 0) {
                const uint32_t stage = c_stage * kStageBytes;
                float s[4][4];                            // four chains of two steps each
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    uint32_t ka[4];
                    ldmatrix4(((k_base + stage) ^ ((ks & 3) << 5)) + (ks >> 2) * 128, ka);
                    if (ks < 4) mma16816_first(s[ks], ka[0], ka[2], ka[1], ka[3], qa[ks][0], qa[ks][1]);
                    else        mma16816(s[ks - 4], ka[0], ka[2], ka[1], ka[3], qa[ks][0], qa[ks][1]);
                }
                uint32_t va[8][4];
                auto load_v = [&](int j) { ldmatrix4_trans(((v_base + stage) ^ ((j & 3) << 5)) + (j >> 2) * 128, va[j]); };
#pragma unroll
                for (int j = 0; j < 4; ++j) load_v(j);
                // this lane's logits: tokens g and g + 8 of its two heads (packed fp32 arithmetic: a pair of heads per instruction)
                auto sum = [&](int k) {
                    return __fmul2_rn(__fadd2_rn(__fadd2_rn(make_float2(s[0][k], s[0][k + 1]), make_float2(s[1][k], s[1][k + 1])),
                                                 __fadd2_rn(make_float2(s[2][k], s[2][k + 1]), make_float2(s[3][k], s[3][k + 1]))), qscale2);
                };
                float2 x = sum(0), y = sum(2);
                if (rows_left < kWarpRows) {
                    if (g >= rows_left) x = make_float2(-INFINITY, -INFINITY);
                    if (g + 8 >= rows_left) y = make_float2(-INFINITY, -INFINITY);
                }
                float2 top = make_float2(fmaxf(x.x, y.x), fmaxf(x.y, y.y)), sc = make_float2(1.f, 1.f);
                if (__any_sync(0xffffffffu, top.x > m.x || top.y > m.y)) {
#pragma unroll
                    for (int d = 4; d < 32; d <<= 1) {
                        top.x = fmaxf(top.x, __shfl_xor_sync(0xffffffffu, top.x, d));
                        top.y = fmaxf(top.y, __shfl_xor_sync(0xffffffffu, top.y, d));
                    }
                    top = make_float2(fmaxf(top.x, m.x), fmaxf(top.y, m.y));
                    sc = make_float2(ex2(m.x - top.x), ex2(m.y - top.y));   // first rows: 2^(-inf) = 0
                    l = __fmul2_rn(l, sc);
                    m = top;
                }
                const float2 neg = make_float2(-m.x, -m.y);
                x = __fadd2_rn(x, neg); y = __fadd2_rn(y, neg);
                x = make_float2(ex2(x.x), ex2(x.y)); y = make_float2(ex2(y.x), ex2(y.y));
                l = __fadd2_rn(l, __fadd2_rn(x, y));
                uint32_t hx, mx, lx, hy, my, ly;
                split_bf16(x, hx, mx, lx);
                split_bf16(y, hy, my, ly);
                float d[8][4];
                if (kFew) {
                    const bool first = qd < 2;            // this lane's columns hold high parts (the others middle ones)
                    const uint32_t hm0 = movmatrix_trans(first ? hx : mx), hm1 = movmatrix_trans(first ? hy : my);
                    const uint32_t lo0 = movmatrix_trans(first ? lx : 0u), lo1 = movmatrix_trans(first ? ly : 0u);
#pragma unroll
                    for (int i = 0; i < 11; ++i) {
                        if (i < 8) {
                            mma16816_first(d[i], va[i][0], va[i][2], va[i][1], va[i][3], hm0, hm1);
                            if (i < 4) load_v(i + 4);
                        }
                        if (i >= 3) { const int j = i - 3; mma16816(d[j], va[j][0], va[j][2], va[j][1], va[j][3], lo0, lo1); }
                    }
                } else {
                    const uint32_t hi0 = movmatrix_trans(hx), hi1 = movmatrix_trans(hy);
                    const uint32_t mi0 = movmatrix_trans(mx), mi1 = movmatrix_trans(my), lo0 = movmatrix_trans(lx), lo1 = movmatrix_trans(ly);
#pragma unroll
                    for (int i = 0; i < 12; ++i) {
                        if (i < 8) {
                            mma16816_first(d[i], va[i][0], va[i][2], va[i][1], va[i][3], hi0, hi1);
                            if (i < 4) load_v(i + 4);
                        }
                        if (i >= 2 && i < 10) { const int j = i - 2; mma16816(d[j], va[j][0], va[j][2], va[j][1], va[j][3], mi0, mi1); }
                        if (i >= 4) { const int j = i - 4; mma16816(d[j], va[j][0], va[j][2], va[j][1], va[j][3], lo0, lo1); }
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    acc[j][0] = __ffma2_rn(acc[j][0], sc, make_float2(d[j][0], d[j][1]));
                    acc[j][1] = __ffma2_rn(acc[j][1], sc, make_float2(d[j][2], d[j][3]));
                }
            }
            if (++c_stage == kStages) c_stage = 0;
        }

        // -------------------------------------------------------------- flush this (CTA, slab) segment
        if (kStep && own_tail && appended && warp == kDecWarps - 1)
            reinterpret_cast<uint4*>(const_cast<uint8_t*>(c_half ? V : K))[new_at] = new_piece;
#pragma unroll
        for (int d = 4; d < 32; d <<= 1) {
            l.x += __shfl_xor_sync(0xffffffffu, l.x, d);
            l.y += __shfl_xor_sync(0xffffffffu, l.y, d);
        }
        if (kFew) {                                       // the same heads' middle parts
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    acc[j][k].x += __shfl_xor_sync(0xffffffffu, acc[j][k].x, 2);
                    acc[j][k].y += __shfl_xor_sync(0xffffffffu, acc[j][k].y, 2);
                }
        }
        if (!kFew || qd < 2) {
            float* wp = wpart + (size_t(warp) * n + 2 * qd) * kWpStride;
            if (2 * qd < n) {
#pragma unroll
                for (int j = 0; j < 8; ++j) { wp[16 * j + g] = acc[j][0].x; wp[16 * j + 8 + g] = acc[j][1].x; }
                if (g == 0) { wp[128] = m.x; wp[129] = l.x; }
            }
            wp += kWpStride;
            if (2 * qd + 1 < n) {
#pragma unroll
                for (int j = 0; j < 8; ++j) { wp[16 * j + g] = acc[j][0].y; wp[16 * j + 8 + g] = acc[j][1].y; }
                if (g == 0) { wp[128] = m.y; wp[129] = l.y; }
            }
        }
        __syncthreads();
        // merge the warps; thread -> channel
        const int fc = int(((long long)(pref[slab] + 1) * Ge - 1) / T), lc = int(((long long)pref[slab + 1] * Ge - 1) / T);
        const int n_part = lc - fc + 1;
        __nv_bfloat16* o = out + (size_t(b) * Hq + size_t(h) * n) * kHeadDim;
        float* rec = dec_part + size_t(cta + slab) * n * kPartStride;
#pragma unroll 1
        for (int hl = 0; hl < n; ++hl) {
            float M = -INFINITY, L = 0.f, A = 0.f;
#pragma unroll
            for (int w = 0; w < kDecWarps; ++w) M = fmaxf(M, wpart[(w * n + hl) * kWpStride + 128]);
#pragma unroll
            for (int w = 0; w < kDecWarps; ++w) {
                const float* p = wpart + (w * n + hl) * kWpStride;
                const float e = ex2(p[128] - M);
                L = fmaf(p[129], e, L);
                A = fmaf(p[tid], e, A);
            }
            if (n_part == 1) {
                o[hl * kHeadDim + tid] = __float2bfloat16_rn(A / L);
            } else {
                rec[hl * kPartStride + tid] = A;
                if (tid == 0) *reinterpret_cast<float2*>(rec + hl * kPartStride + 128) = make_float2(M, L);
            }
        }
        __syncthreads();                                   // every thread's record stores are ordered before the arrival; wpart is free
        if (n_part > 1) {
            if (tid == 0) {
                const uint32_t old = arrive_acq_rel(dec_cnt + slab);
                const int last = (old == uint32_t(n_part - 1)) ? 1 : 0;
                if (last) dec_cnt[slab] = 0u;              // self-resetting for the next launch
                s_last = last;
            }
            __syncthreads();
            if (s_last) {
                // The launch waits for this merge, so all its loads go out together: a warp takes a head, a lane a partial
                // for the weights (max, sum) and four channels for the accumulators, the first kAhead of which are
                // requested before the weights are known.  (In rounds of four behind the weights, 18 partials took 7 us.  With 20 ahead a
                // step of one sequence takes 281 us instead of 285, but two of 80 slabs with three partials each 74.9 instead of 72.9: the
                // code is fetched for the first time in the launch, and every instruction of it counts.)
                const float* r0 = dec_part + size_t(fc + slab) * n * kPartStride;
                constexpr int kAhead = kFew ? 10 : 12;
                const int stride = n * kPartStride;
#pragma unroll 1
                for (int hl = warp; hl < n; hl += kDecWarps) {
                    const float* rh = r0 + hl * kPartStride;
                    auto channels = [&](int p) { return __ldcg(reinterpret_cast<const float4*>(rh + size_t(p * stride)) + lane); };
                    float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
                    float M = -INFINITY, L = 0.f;
#pragma unroll 1
                    for (int p0 = 0; p0 < n_part; p0 += 32) {
                        const float2 ml = __ldcg(reinterpret_cast<const float2*>(rh + size_t(min(p0 + lane, n_part - 1) * stride) + 128));
                        float4 a[kAhead];
#pragma unroll
                        for (int k = 0; k < kAhead; ++k)
                            if (p0 + k < n_part) a[k] = channels(p0 + k);
                        const bool on = p0 + lane < n_part;
                        float mx = on ? ml.x : -INFINITY;
#pragma unroll
                        for (int d = 16; d; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
                        const float Mn = fmaxf(M, mx), keep = ex2(M - Mn);          // first round: 2^(-inf) = 0
                        const float w = on ? ex2(ml.x - Mn) : 0.f;
                        float ls = on ? ml.y * w : 0.f;
#pragma unroll
                        for (int d = 16; d; d >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, d);
                        L = fmaf(L, keep, ls);
                        M = Mn;
                        A.x *= keep; A.y *= keep; A.z *= keep; A.w *= keep;
                        const int cnt = min(32, n_part - p0);
#pragma unroll 1
                        for (int k0 = 0; k0 < cnt; k0 += kAhead) {
#pragma unroll
                            for (int k = 0; k < kAhead; ++k) {
                                if (k0 + k < cnt) {
                                    const float wk = __shfl_sync(0xffffffffu, w, k0 + k);
                                    A.x = fmaf(a[k].x, wk, A.x); A.y = fmaf(a[k].y, wk, A.y);
                                    A.z = fmaf(a[k].z, wk, A.z); A.w = fmaf(a[k].w, wk, A.w);
                                }
                            }
                            if (k0 + kAhead < cnt) {
#pragma unroll
                                for (int k = 0; k < kAhead; ++k)
                                    if (k0 + kAhead + k < cnt) a[k] = channels(p0 + k0 + kAhead + k);
                            }
                        }
                    }
                    const float inv = 1.f / L;
                    __nv_bfloat16* oi = o + hl * kHeadDim + lane * 4;
                    oi[0] = __float2bfloat16_rn(A.x * inv); oi[1] = __float2bfloat16_rn(A.y * inv);
                    oi[2] = __float2bfloat16_rn(A.z * inv); oi[3] = __float2bfloat16_rn(A.w * inv);
                }
            }
        }
        if (own_tail) step_tables(slab, b, n_rows, appended, step_S0, step_starts);
    }
    cp_async_wait<0>();
    if (!triggered) pdl_trigger();
    // slabs with no row to attend to: zeros (owned round-robin); in the fused step they have no room: unchanged, reported
#pragma unroll 1
    for (int s = cta; s < n_slabs; s += G) {
        if (lens[s] >> 1) continue;
        const int b = s / Hk, h = s % Hk;
        __nv_bfloat16* o = out + (size_t(b) * Hq + size_t(h) * n) * kHeadDim;
#pragma unroll 1
        for (int idx = tid; idx < n * kHeadDim; idx += kDecThreads) o[idx] = __float2bfloat16_rn(0.f);
        if (kStep) step_tables(s, b, 0, false, 0, 0);
    }
}

}  // namespace skipkv

using namespace skipkv;

static size_t dec_smem_bytes(int slabs, int group) {
    return size_t(kRingBytes) + size_t(kDecWarps) * group * kWpStride * 4 + size_t(2 * slabs + 1) * 4;
}

static int decode_impl(const skipkv_shape* shape, const void* q, const void* K, const void* V, const int32_t* kv_len,
                       void* out, void* hidden, const void* steer_vec, const float* alpha, const uint8_t* flag,
                       const int32_t* block_table, int max_pages, const StepArgs& step, void* ws, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!q || !K || !V || !kv_len || !out) return SKIPKV_ERR_INVALID_ARG;
    if (hidden && (!steer_vec || !alpha || !flag || shape->d_model <= 0)) return SKIPKV_ERR_INVALID_ARG;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return SKIPKV_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(K) & 15) || (reinterpret_cast<uintptr_t>(V) & 15) ||
        (reinterpret_cast<uintptr_t>(q) & 15))
        return SKIPKV_ERR_INVALID_ARG;
    const WsLayout L = make_layout(*shape);
    if (L.slabs > kMaxDecSlabs) return SKIPKV_ERR_UNSUPPORTED;
    uint8_t* w = static_cast<uint8_t*>(ws);
    const size_t smem = dec_smem_bytes(L.slabs, L.group);
    if (smem > 227 * 1024) {                         // the per-slab tile table no longer fits beside the tile ring
        set_error_text("skipkv_decode_attn: batch * n_kv_heads too large for the shared-memory tile table");
        return SKIPKV_ERR_UNSUPPORTED;
    }
    const int grid = num_sms() < kDecMaxGrid ? num_sms() : kDecMaxGrid;
    SKIPKV_CUDA(launch_dependent(
        L.group <= 4 ? (step.k_new ? decode_attn_kernel<true, true> : decode_attn_kernel<false, true>)
                     : (step.k_new ? decode_attn_kernel<true, false> : decode_attn_kernel<false, false>), dim3(grid), dim3(kDecThreads), smem,
        static_cast<cudaStream_t>(stream), int(shape->batch), int(shape->n_q_heads), int(shape->n_kv_heads), int(L.slabs),
        static_cast<long long>(shape->total_rows), shape->slab_off, shape->cap, static_cast<const __nv_bfloat16*>(q),
        static_cast<const uint8_t*>(K), static_cast<const uint8_t*>(V), kv_len, static_cast<__nv_bfloat16*>(out),
        &reinterpret_cast<Header*>(w + L.header)->status, reinterpret_cast<uint32_t*>(w + L.dec_cnt),
        reinterpret_cast<float*>(w + L.dec_part), int(shape->d_model), static_cast<__nv_bfloat16*>(hidden),
        static_cast<const __nv_bfloat16*>(steer_vec), alpha, flag, block_table, max_pages, step));
    return SKIPKV_OK;
}

extern "C" int skipkv_decode_attn(const skipkv_shape* shape, const void* q, const void* K, const void* V,
                                  const int32_t* kv_len, void* out, void* hidden, const void* steer_vec,
                                  const float* alpha, const uint8_t* flag, void* ws, void* stream) {
    return decode_impl(shape, q, K, V, kv_len, out, hidden, steer_vec, alpha, flag, nullptr, 0, StepArgs{}, ws, stream);
}

extern "C" int skipkv_decode_attn_paged(const skipkv_shape* shape, const void* q, const void* K_pages,
                                        const void* V_pages, const int32_t* block_table, int32_t max_pages,
                                        const int32_t* kv_len, void* out, void* hidden, const void* steer_vec,
                                        const float* alpha, const uint8_t* flag, void* ws, void* stream) {
    if (!block_table || max_pages <= 0) return SKIPKV_ERR_INVALID_ARG;
    return decode_impl(shape, q, K_pages, V_pages, kv_len, out, hidden, steer_vec, alpha, flag, block_table, max_pages,
                       StepArgs{}, ws, stream);
}

extern "C" int skipkv_decode_step(const skipkv_shape* shape, const void* q, const void* k_new, const void* v_new, void* K,
                                  void* V, const int32_t* kv_len_in, int32_t* kv_len_out, int32_t* sent_off,
                                  int32_t* sent_id, int32_t* n_sent, const uint8_t* new_sent, const int32_t* gen_id,
                                  void* q_win, int32_t slot, void* out, void* hidden, const void* steer_vec,
                                  const float* alpha, const uint8_t* flag, void* ws, void* stream) {
    if (!k_new || !v_new || !kv_len_in || !kv_len_out || kv_len_in == kv_len_out || !sent_off || !sent_id || !n_sent ||
        !new_sent || !gen_id)
        return SKIPKV_ERR_INVALID_ARG;
    if (int rc = check_shape(shape)) return rc;
    if (shape->max_sent <= 0) return SKIPKV_ERR_INVALID_ARG;
    if (q_win && (slot < 0 || slot >= shape->window)) return SKIPKV_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(k_new) | reinterpret_cast<uintptr_t>(v_new) | reinterpret_cast<uintptr_t>(q_win)) & 15)
        return SKIPKV_ERR_INVALID_ARG;
    StepArgs step{};
    step.k_new = static_cast<const uint4*>(k_new); step.v_new = static_cast<const uint4*>(v_new);
    step.kv_len_out = kv_len_out; step.sent_off = sent_off; step.sent_id = sent_id; step.n_sent = n_sent;
    step.new_sent = new_sent; step.gen_id = gen_id; step.q_win = static_cast<uint4*>(q_win);
    step.window = shape->window; step.slot = slot; step.max_sent = shape->max_sent;
    return decode_impl(shape, q, K, V, kv_len_in, out, hidden, steer_vec, alpha, flag, nullptr, 0, step, ws, stream);
}

extern "C" int skipkv_decode_step_paged(const skipkv_shape* shape, const void* q, const void* k_new, const void* v_new,
                                        void* K_pages, void* V_pages, const int32_t* block_table, int32_t max_pages,
                                        const int32_t* kv_len_in, int32_t* kv_len_out, int32_t* sent_off, int32_t* sent_id,
                                        int32_t* n_sent, const uint8_t* new_sent, const int32_t* gen_id, void* q_win,
                                        int32_t slot, void* out, void* hidden, const void* steer_vec, const float* alpha,
                                        const uint8_t* flag, void* ws, void* stream) {
    if (!block_table || max_pages <= 0) return SKIPKV_ERR_INVALID_ARG;
    if (!k_new || !v_new || !kv_len_in || !kv_len_out || kv_len_in == kv_len_out || !sent_off || !sent_id || !n_sent ||
        !new_sent || !gen_id)
        return SKIPKV_ERR_INVALID_ARG;
    if (int rc = check_shape(shape)) return rc;
    if (shape->max_sent <= 0) return SKIPKV_ERR_INVALID_ARG;
    if (q_win && (slot < 0 || slot >= shape->window)) return SKIPKV_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(k_new) | reinterpret_cast<uintptr_t>(v_new) | reinterpret_cast<uintptr_t>(q_win)) & 15)
        return SKIPKV_ERR_INVALID_ARG;
    StepArgs step{};
    step.k_new = static_cast<const uint4*>(k_new); step.v_new = static_cast<const uint4*>(v_new);
    step.kv_len_out = kv_len_out; step.sent_off = sent_off; step.sent_id = sent_id; step.n_sent = n_sent;
    step.new_sent = new_sent; step.gen_id = gen_id; step.q_win = static_cast<uint4*>(q_win);
    step.window = shape->window; step.slot = slot; step.max_sent = shape->max_sent;
    return decode_impl(shape, q, K_pages, V_pages, kv_len_in, out, hidden, steer_vec, alpha, flag, block_table, max_pages, step,
                       ws, stream);
}

// ---------------------------------------------------------------------------------------------
// Decode attention for callers that cannot provide a workspace.
//
// Some callers have no device allocator to draw scratch from: a serving process that handed every
// free byte of HBM to its KV-cache pool at start-up (so a later cudaMalloc would fail), or a
// plug-in that is forbidden to allocate because cudaMalloc synchronises the whole device and would
// stall the other streams of the process.  For them the partial results and arrival counters of
// the kernel live in the fixed array below, which every GPU that loads this library holds until
// the process exits (about 2 MB).  Sizes are therefore capped: at most SKIPKV_STATIC_MAX_SLABS
// (sequence, head) slabs and a decode grid of at most kStaticMaxCtas CTAs.
//
// The array's name is only a host-side handle in host code; the device address is looked up once
// per device with cudaGetSymbolAddress (with that device current) and handed to the kernel.
// ---------------------------------------------------------------------------------------------
namespace skipkv {

constexpr int kStaticMaxSlabs = SKIPKV_STATIC_MAX_SLABS;
constexpr int kStaticMaxCtas = kDecMaxGrid;
constexpr size_t kStaticCntOff = 256;                                      // after the status word
constexpr size_t kStaticPartOff = kStaticCntOff + size_t(kStaticMaxSlabs) * 4;
constexpr size_t kStaticBytes =
    kStaticPartOff + size_t(kStaticMaxCtas + kStaticMaxSlabs) * kMaxGroup * kPartStride * 4;

static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

// The array keeps whatever the previous call left: the status word and the arrival counters must start at zero (the partial records
// are fully written before they are read).  A kernel and not a memset, so that decode attention, as its programmatic dependent, derives its
// schedule meanwhile.
__global__ void __launch_bounds__(256) static_clear_kernel(uint32_t* words) {
    pdl_trigger();
    pdl_wait();
    for (int i = threadIdx.x; i < int(kStaticPartOff / 4); i += 256) words[i] = 0u;
}

constexpr int kMaxDevices = 64;
static unsigned char* g_static_addr[kMaxDevices];      // device address of the array, per device
static bool g_static_ready[kMaxDevices];
static std::mutex g_static_mutex;

// First call on a device: resolve the array's device address.  Later calls only read the cached pointer.
static int static_setup(int dev, unsigned char** base) {
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ready[dev]) {
        void* p = nullptr;
        SKIPKV_CUDA(cudaGetSymbolAddress(&p, g_static_scratch));
        if (!p) return SKIPKV_ERR_CUDA;
        g_static_addr[dev] = static_cast<unsigned char*>(p);
        g_static_ready[dev] = true;
    }
    *base = g_static_addr[dev];
    return SKIPKV_OK;
}

}  // namespace skipkv

extern "C" int skipkv_decode_attn_static(const skipkv_shape* shape, const void* q, const void* K, const void* V,
                                         const int32_t* kv_len, void* out, void* hidden, const void* steer_vec,
                                         const float* alpha, const uint8_t* flag, uint32_t* status, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!q || !K || !V || !kv_len || !out) return SKIPKV_ERR_INVALID_ARG;
    if (hidden && (!steer_vec || !alpha || !flag || shape->d_model <= 0)) return SKIPKV_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(K) & 15) || (reinterpret_cast<uintptr_t>(V) & 15) ||
        (reinterpret_cast<uintptr_t>(q) & 15))
        return SKIPKV_ERR_INVALID_ARG;
    const int slabs = shape->batch * shape->n_kv_heads;
    if (slabs > kStaticMaxSlabs) {
        char msg[160];
        std::snprintf(msg, sizeof(msg),
                      "skipkv_decode_attn_static: batch*n_kv_heads = %d exceeds SKIPKV_STATIC_MAX_SLABS = %d; "
                      "use skipkv_decode_attn with a workspace",
                      slabs, kStaticMaxSlabs);
        set_error_text(msg);
        return SKIPKV_ERR_UNSUPPORTED;
    }
    int dev = 0;
    SKIPKV_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) {
        set_error_text("skipkv_decode_attn_static: device ordinal beyond 63");
        return SKIPKV_ERR_UNSUPPORTED;
    }
    const size_t smem = dec_smem_bytes(slabs, shape->n_q_heads / shape->n_kv_heads);
    unsigned char* base = nullptr;
    if (int rc = static_setup(dev, &base)) return rc;
    const auto kernel = shape->n_q_heads / shape->n_kv_heads <= 4 ? decode_attn_kernel<false, true> : decode_attn_kernel<false, false>;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SKIPKV_CUDA(launch_dependent(static_clear_kernel, dim3(1), dim3(256), 0, st, reinterpret_cast<uint32_t*>(base)));
    const int grid = num_sms() < kStaticMaxCtas ? num_sms() : kStaticMaxCtas;
    uint32_t* status_word = status ? status : reinterpret_cast<uint32_t*>(base);
    SKIPKV_CUDA(launch_dependent(
        kernel, dim3(grid), dim3(kDecThreads), smem, st, int(shape->batch), int(shape->n_q_heads), int(shape->n_kv_heads), slabs,
        static_cast<long long>(shape->total_rows), shape->slab_off, shape->cap, static_cast<const __nv_bfloat16*>(q),
        static_cast<const uint8_t*>(K), static_cast<const uint8_t*>(V), kv_len, static_cast<__nv_bfloat16*>(out), status_word,
        reinterpret_cast<uint32_t*>(base + kStaticCntOff), reinterpret_cast<float*>(base + kStaticPartOff), int(shape->d_model),
        static_cast<__nv_bfloat16*>(hidden), static_cast<const __nv_bfloat16*>(steer_vec), alpha, flag,
        static_cast<const int32_t*>(nullptr), 0, StepArgs{}));
    return SKIPKV_OK;
}
