// skipkv_select: which sentences survive under the KV budget (paper Section 4.1: evict in
// increasing order of the final score until the cache meets budget B), at sentence granularity.
//
// One CTA per (sequence, head) slab.  The ranking is: protected-tail sentences in index order, then the rest by score
// descending with ties broken by the lower index (exact fp32 comparison, -0 == +0); a sentence survives iff its inclusive
// running total of lengths in rank order is within the budget.  Lengths are non-negative, so the total is monotone and
// this is exactly "the longest rank prefix that fits; stop at the first sentence that does not": nothing has to be sorted,
// only the score has to be found at which the total crosses the budget.  It is found digit by digit (8 bits at a time,
// from the top): a histogram of lengths over the sentences that share the digits so far, and the bin in which the
// running total crosses; sentences of exactly that score are then taken in index order.  One barrier per digit (every warp
// scans the histogram itself).  A bitonic sort of 1024 keys took 55 rounds and 14 us per call; this takes 4 digits.
// skipkv_select_fill then lets the first sentence that does not fit keep its most important tokens, so that exactly B survive.
#include "common.cuh"

namespace skipkv {

constexpr int kSelThreads = 512;

__device__ __forceinline__ uint32_t orderable(float f) {
    uint32_t u = __float_as_uint(f);
    if ((u << 1) == 0u) u = 0u;                        // -0 -> +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u); // ascending in f
}

// each thread passes its local total, gets the exclusive offset of its first element
__device__ __forceinline__ uint32_t block_excl(uint32_t v, uint32_t* wsum, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t a = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += a;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    const uint32_t w = lane < kSelThreads / 32 ? wsum[lane] : 0u;
    uint32_t base = lane < warp ? w : 0u, t = w;
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        base += __shfl_xor_sync(0xffffffffu, base, d);
        t += __shfl_xor_sync(0xffffffffu, t, d);
    }
    total = t;
    __syncthreads();
    return base + inc - v;
}

// Exactly-B retention: where tok_keep is non-null the first sentence that does not fit keeps its `slack` tokens of
// largest importance (equal values: the earlier token), flagged in tok_keep (one byte per cache row), and gets
// keep = 2.  tok_imp is indexed by cache row when from_rows is set, else [slab][max_cap].
struct FillArgs {
    const float* tok_imp;
    const float* tok_red;      // nullable, one value per cache row: the cut sentence's tokens are then ordered by
    float sigma;               // sigma * tok_imp - (1 - sigma) * tok_red (each operation rounded to fp32)
    uint8_t* tok_keep;
    const int64_t* slab_off;
    const int32_t* cap;
    int Hk, max_cap, from_rows;
};

constexpr int kSelAhead = 2;            // sentences per thread that are read before their number is known
constexpr int kFillStage = 1024;        // tokens of a cut sentence whose order keys are staged in shared memory

__global__ void __launch_bounds__(kSelThreads)
select_kernel(int max_sent, int budget, int protect_tail, const float* sent_score, const int32_t* sent_off,
              const int32_t* n_sent, uint8_t* keep, int32_t* kept_idx, int32_t* n_kept, int32_t* new_len,
              FillArgs fill, uint32_t* status) {
    extern __shared__ __align__(16) uint8_t sel_smem[];
    uint32_t* keys = reinterpret_cast<uint32_t*>(sel_smem);            // [max_sent] ascending in rank; a thread touches its own only
    int* lens = reinterpret_cast<int*>(keys + max_sent);               // [max_sent] length, negative - 1 if protected
    __shared__ uint32_t hist[4][256], wsum[kSelThreads / 32];
    __shared__ uint32_t s_forced;
    __shared__ int s_cut, s_slack, s_begin, s_total;
    __shared__ float s_key[kFillStage];
    pdl_trigger();
    const int slab = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < 4 * 256; i += kSelThreads) (&hist[0][0])[i] = 0u;
    if (tid == 0) { s_forced = 0u; s_cut = -1; s_slack = 0; s_total = 0; }
    pdl_wait();                                          // inputs may come from the kernel before
    const float* score = sent_score + size_t(slab) * max_sent;
    const int32_t* so = sent_off + size_t(slab) * (max_sent + 1);
    uint8_t* kp = keep + size_t(slab) * max_sent;
    int32_t* ki = kept_idx ? kept_idx + size_t(slab) * max_sent : nullptr;
    // The kernel is a chain of round trips to memory, so everything is requested at once where the table is small enough for a fixed share of
    // it per thread: the shares (whatever is in them past the last sentence), the number of sentences and the slab's first row.
    const bool ahead = max_sent <= kSelAhead * kSelThreads;
    const int per_max = (max_sent + kSelThreads - 1) / kSelThreads;
    int off[kSelAhead + 1];
    float sc[kSelAhead];
#pragma unroll
    for (int q = 0; q <= kSelAhead; ++q) {
        const int i = tid * per_max + q;
        off[q] = ahead && q <= per_max && i <= max_sent ? so[i] : 0;
        if (q < kSelAhead) sc[q] = ahead && q < per_max && i < max_sent ? score[i] : 0.f;
    }
    const size_t row0 = fill.tok_keep ? slab_row0(fill.slab_off, fill.cap, fill.Hk, slab / fill.Hk, slab % fill.Hk) : 0;
    int S = n_sent[slab];
    if (S < 0 || S > max_sent) {
        if (tid == 0) atomicOr(status, SKIPKV_STATUS_BAD_TABLE);
        S = 0;
    }
    const int per = ahead ? per_max : (S + kSelThreads - 1) / kSelThreads;
    const int i0 = min(tid * per, S), i1 = min(i0 + per, S);   // this thread's sentences
    if (ahead) {
#pragma unroll
        for (int q = 0; q < kSelAhead; ++q)
            if (i0 + q == S - 1 && i0 + q < i1) s_total = off[q + 1];
    } else if (tid == 0 && S > 0) {
        s_total = so[S];
    }
    __syncthreads();                                     // the total is known, the histograms are clear
    const int total = s_total;

    if (total <= budget) {                              // already fits: identity
        for (int i = tid; i < max_sent; i += kSelThreads) {
            kp[i] = (i < S) ? 1 : 0;
            if (ki) ki[i] = (i < S) ? i : -1;
        }
        if (tid == 0) {
            if (n_kept) n_kept[slab] = S;
            if (new_len) new_len[slab] = total;
        }
        return;
    }

    auto take = [&](int i, int b, int e, float x) {
        const bool forced = protect_tail > 0 && e > total - protect_tail && e > b;
        const uint32_t k = ~orderable(x);
        keys[i] = k;
        lens[i] = forced ? -(e - b) - 1 : e - b;
        if (forced) atomicAdd(&s_forced, uint32_t(e - b));
        else if (e > b) atomicAdd(&hist[0][k >> 24], uint32_t(e - b));
    };
    if (ahead) {
#pragma unroll
        for (int q = 0; q < kSelAhead; ++q)
            if (i0 + q < i1) take(i0 + q, off[q], off[q + 1], sc[q]);
    } else {
        for (int i = i0; i < i1; ++i) take(i, so[i], so[i + 1], score[i]);
    }
    __syncthreads();
    const uint32_t forced_len = s_forced;
    const bool only_forced = forced_len > uint32_t(budget);      // then the protected sentences alone, in index order
    uint32_t room = only_forced ? uint32_t(budget) : uint32_t(budget) - forced_len;    // left for the sentences of score `cross`
    uint32_t cross = 0;
    if (!only_forced) {
#pragma unroll 1
        for (int d = 0; d < 4; ++d) {
            // bin in which the running total exceeds the room: 8 bins per lane, every warp for itself
            const int shift = 24 - 8 * d;
            uint32_t h[8], mine = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) { h[q] = hist[d][lane * 8 + q]; mine += h[q]; }
            uint32_t inc = mine;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const uint32_t x = __shfl_up_sync(0xffffffffu, inc, s);
                if (lane >= s) inc += x;
            }
            const int src = __ffs(__ballot_sync(0xffffffffu, inc > room)) - 1;     // (the total exceeds the room: some lane's does)
            uint32_t before = inc - mine, bin = uint32_t(lane) * 8u;
#pragma unroll
            for (int q = 0; q < 7; ++q)
                if (before + h[q] <= room && bin == uint32_t(lane) * 8u + q) { before += h[q]; ++bin; }
            bin = __shfl_sync(0xffffffffu, bin, src);
            room -= __shfl_sync(0xffffffffu, before, src);
            cross |= bin << shift;
            if (d < 3) {
                for (int i = i0; i < i1; ++i)
                    if (lens[i] > 0 && ((keys[i] ^ cross) >> shift) == 0u) atomicAdd(&hist[d + 1][(keys[i] >> (shift - 8)) & 255u], uint32_t(lens[i]));
                __syncthreads();
            }
        }
    }
    // sentences at the crossing are taken in index order; the first of them that does not fit is the cut one
    auto at_cross = [&](int i) { return only_forced ? lens[i] < 0 : (lens[i] >= 0 && keys[i] == cross); };
    auto length = [&](int i) { return uint32_t(lens[i] < 0 ? -lens[i] - 1 : lens[i]); };
    uint32_t local = 0, all;
    for (int i = i0; i < i1; ++i) local += at_cross(i) ? length(i) : 0u;
    uint32_t run = block_excl(local, wsum, all);
    uint32_t cnt = 0, kept_tokens = 0;
    for (int i = i0; i < i1; ++i) {
        bool k;
        if (at_cross(i)) {
            const uint32_t before = run;
            run += length(i);
            k = run <= room;
            if (!k && before < room) {                   // one sentence only
                s_cut = i; s_slack = int(room - before);
                s_begin = !ahead ? so[i] : i == i0 ? off[0] : off[1];
            }
        } else {
            k = !only_forced && (lens[i] < 0 || keys[i] < cross);
        }
        kept_tokens += k ? length(i) : 0u;
        keys[i] = k ? 1u : 0u;
    }
    uint32_t sum_tokens;
    block_excl(kept_tokens, wsum, sum_tokens);           // (its barriers also publish the cut)
    const bool filled = fill.tok_keep && s_cut >= 0;
    if (filled) {
        const int c = s_cut, slack = s_slack;
        const int cb = s_begin, len = int(length(c));
        const float* imp = fill.from_rows ? fill.tok_imp + row0 + cb : fill.tok_imp + size_t(slab) * fill.max_cap + cb;
        uint8_t* tk = fill.tok_keep + row0 + cb;
        const float* red = fill.tok_red ? fill.tok_red + row0 + cb : nullptr;
        const float w_red = __fsub_rn(1.f, fill.sigma);
        auto key = [&](int u) {
            const float i = __ldg(imp + u);
            return red ? __fsub_rn(__fmul_rn(fill.sigma, i), __fmul_rn(w_red, __ldg(red + u))) : i;
        };
        const bool staged = len <= kFillStage;
        if (staged) {
            for (int u = tid; u < len; u += kSelThreads) s_key[u] = key(u);
            __syncthreads();
        }
        for (int t = tid; t < len; t += kSelThreads) {   // rank by counting: tokens that come before t in the order
            const float mine = staged ? s_key[t] : key(t);
            int rank = 0;
            if (staged) {
#pragma unroll 8
                for (int u = 0; u < len; ++u) { const float other = s_key[u]; rank += (other > mine || (other == mine && u < t)) ? 1 : 0; }
            } else {
                for (int u = 0; u < len; ++u) { const float other = key(u); rank += (other > mine || (other == mine && u < t)) ? 1 : 0; }
            }
            tk[t] = rank < slack ? 1 : 0;
        }
    }
    // outputs in sentence-index order
    for (int i = i0; i < i1; ++i) cnt += (keys[i] || (filled && i == s_cut)) ? 1u : 0u;
    uint32_t nk;
    uint32_t pos = block_excl(cnt, wsum, nk);
    for (int i = i0; i < i1; ++i) {
        const uint8_t f = keys[i] ? 1 : (filled && i == s_cut ? 2 : 0);
        kp[i] = f;
        if (f && ki) ki[pos] = i;
        pos += f ? 1u : 0u;
    }
    for (int i = S + tid; i < max_sent; i += kSelThreads) kp[i] = 0;
    if (ki) for (int i = int(nk) + tid; i < max_sent; i += kSelThreads) ki[i] = -1;
    if (tid == 0) {
        if (n_kept) n_kept[slab] = int(nk);
        if (new_len) new_len[slab] = filled ? budget : int(sum_tokens);
    }
}

}  // namespace skipkv

using namespace skipkv;

static int select_impl(const skipkv_shape* shape, const skipkv_params* params, const float* sent_score,
                       const int32_t* sent_off, const int32_t* n_sent, uint8_t* keep, int32_t* kept_idx,
                       int32_t* n_kept, int32_t* new_len, FillArgs fill, void* ws, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!params || !sent_score || !sent_off || !n_sent || !keep) return SKIPKV_ERR_INVALID_ARG;
    if (params->budget < 0 || params->protect_tail < 0) return SKIPKV_ERR_INVALID_ARG;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return SKIPKV_ERR_WORKSPACE;
    const size_t smem = size_t(shape->max_sent) * 8;
    if (shape->max_sent > 16384) return SKIPKV_ERR_UNSUPPORTED;
    const int slabs = shape->batch * shape->n_kv_heads;
    SKIPKV_CUDA(launch_dependent(select_kernel, dim3(slabs), dim3(kSelThreads), smem, static_cast<cudaStream_t>(stream),
                                 shape->max_sent, params->budget, params->protect_tail, sent_score, sent_off, n_sent, keep,
                                 kept_idx, n_kept, new_len, fill, &static_cast<Header*>(ws)->status));
    return SKIPKV_OK;
}

extern "C" int skipkv_select(const skipkv_shape* shape, const skipkv_params* params, const float* sent_score,
                             const int32_t* sent_off, const int32_t* n_sent, uint8_t* keep, int32_t* kept_idx,
                             int32_t* n_kept, int32_t* new_len, void* ws, void* stream) {
    return select_impl(shape, params, sent_score, sent_off, n_sent, keep, kept_idx, n_kept, new_len, FillArgs{}, ws,
                       stream);
}

static int select_fill_impl(const skipkv_shape* shape, const skipkv_params* params, const float* sent_score,
                            const float* tok_imp, const float* tok_red, const int32_t* sent_off, const int32_t* n_sent,
                            uint8_t* keep, uint8_t* tok_keep, int32_t* kept_idx, int32_t* n_kept, int32_t* new_len, void* ws,
                            void* stream) {
    if (!tok_keep || !params) return SKIPKV_ERR_INVALID_ARG;
    if (int rc = check_shape(shape)) return rc;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return SKIPKV_ERR_WORKSPACE;
    FillArgs fill{};
    fill.tok_keep = tok_keep;
    fill.tok_red = tok_red;
    fill.sigma = params->sigma;
    fill.slab_off = shape->slab_off; fill.cap = shape->cap; fill.Hk = shape->n_kv_heads; fill.max_cap = shape->max_cap;
    if (tok_imp) { fill.tok_imp = tok_imp; fill.from_rows = 1; }
    else { fill.tok_imp = reinterpret_cast<const float*>(static_cast<uint8_t*>(ws) + make_layout(*shape).sc_tokimp); }
    return select_impl(shape, params, sent_score, sent_off, n_sent, keep, kept_idx, n_kept, new_len, fill, ws, stream);
}

extern "C" int skipkv_select_fill(const skipkv_shape* shape, const skipkv_params* params, const float* sent_score,
                                  const float* tok_imp, const int32_t* sent_off, const int32_t* n_sent, uint8_t* keep,
                                  uint8_t* tok_keep, int32_t* kept_idx, int32_t* n_kept, int32_t* new_len, void* ws,
                                  void* stream) {
    return select_fill_impl(shape, params, sent_score, tok_imp, nullptr, sent_off, n_sent, keep, tok_keep, kept_idx, n_kept,
                            new_len, ws, stream);
}

extern "C" int skipkv_select_fill_red(const skipkv_shape* shape, const skipkv_params* params, const float* sent_score,
                                      const float* tok_imp, const float* tok_red, const int32_t* sent_off,
                                      const int32_t* n_sent, uint8_t* keep, uint8_t* tok_keep, int32_t* kept_idx,
                                      int32_t* n_kept, int32_t* new_len, void* ws, void* stream) {
    if (!tok_red) return SKIPKV_ERR_INVALID_ARG;
    return select_fill_impl(shape, params, sent_score, tok_imp, tok_red, sent_off, n_sent, keep, tok_keep, kept_idx, n_kept,
                            new_len, ws, stream);
}
