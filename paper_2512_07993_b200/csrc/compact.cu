// skipkv_compact: in-place stream compaction of the surviving K/V rows (paper Algorithm 1,
// eviction + post-eviction range update, Eq. "after").
//
// Two launches on the caller's stream:
//   plan  one CTA per (sequence, head) slab.  Block-wide scans over the keep flags turn the
//         sentence table into (a) the rewritten tables, (b) a list of runs: maximal groups
//         of adjacent kept sentences, each a contiguous source block that lands on a
//         contiguous destination block, and (c) for every segment of kSegRows destination rows
//         the run it starts in and the destination of the survivors that lie in its way.
//   move  persistent CTAs.  K and V of a slab are two independent streams; a stream's
//         destination range is cut into segments which are handed out in ascending order by
//         an atomic ticket.  A CTA pulls every source piece of its segment into shared memory
//         with bulk asynchronous copies (one copy per run piece, no register staging), flags
//         "segment j of this stream is loaded", and then writes the pieces to their
//         destination with bulk stores.
//
// With partly kept sentences (skipkv_compact_fill: keep == 2, survivors flagged per token) the plan first packs
// the surviving rows of such a sentence to the front of the sentence's own rows, so that it becomes a shorter
// contiguous sentence (a run of its own, whose index-map entries the plan writes) and the move proceeds unchanged.
//
// Why this is safe in place: rows only move down (dst <= src), so a store into segment j can
// only overwrite source rows of segments <= j, and of those only the rows that lie inside segment j itself: survivors
// seg_dep[j] .. seg_dep[j+1] of the destination order, which are at most kSegRows and so belong to one or two segments.  A
// segment stores after its own loads have landed and after those segments have flagged theirs.  Tickets are issued in
// ascending segment order, so whatever a CTA waits for is already held by a CTA that runs, and the lowest segment
// not yet loaded waits for nothing: the wait cannot deadlock, and it is bounded anyway (on expiry the status
// word is flagged and the stores of that segment are skipped).
//
// The move is bound by DRAM (every kept row is read and written once).  32 KB segments, six CTAs to an SM: the pieces
// of the last round are small, and a CTA draws its next ticket while it works on the present one, reads what the plan
// knows of a segment in two rounds of independent loads, and waits for one or two flags instead of for all lower
// segments in turn.  With 64 KB segments, three CTAs to an SM, a search for the first run and a counter that every segment of
// a stream had to pass in order the move took 65 us; now it takes 62 (80 slabs x 4.1K kept rows of 24K: 5.4 TB/s), the whole
// call with the selection 79 instead of 87.
#include "common.cuh"

namespace skipkv {

constexpr int kSegBytes = kSegRows * kRowBytes;
constexpr int kMoveThreads = 64;                    // a warp for the copies, one for the index map
constexpr int kMoveCtas = 6;                        // per SM: what the shared memory holds
constexpr int kPlanThreads = 1024;

// exclusive block scan of three ints at once; returns the block totals through tot[]
__device__ __forceinline__ void block_scan3(int v0, int v1, int v2, int& e0, int& e1, int& e2, int tot[3],
                                            int (*wsum)[3]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int i0 = v0, i1 = v1, i2 = v2;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int a0 = __shfl_up_sync(0xffffffffu, i0, d), a1 = __shfl_up_sync(0xffffffffu, i1, d),
                  a2 = __shfl_up_sync(0xffffffffu, i2, d);
        if (lane >= d) { i0 += a0; i1 += a1; i2 += a2; }
    }
    if (lane == 31) { wsum[warp][0] = i0; wsum[warp][1] = i1; wsum[warp][2] = i2; }
    __syncthreads();
    int b0 = 0, b1 = 0, b2 = 0, t0 = 0, t1 = 0, t2 = 0;
    for (int w = 0; w < nw; ++w) {
        if (w == warp) { b0 = t0; b1 = t1; b2 = t2; }
        t0 += wsum[w][0]; t1 += wsum[w][1]; t2 += wsum[w][2];
    }
    e0 = b0 + i0 - v0; e1 = b1 + i1 - v1; e2 = b2 + i2 - v2;
    tot[0] = t0; tot[1] = t1; tot[2] = t2;
    __syncthreads();
}

// Rows of tokens [pb, pe) of a slab whose flag is set move, in order, to rows pb, pb+1, ... of the same slab; survivor k came from
// token map[k].  K and V together, 128 rows per pass: every thread holds two 16-byte pieces of each; all pieces of a pass are read before any
// is written, and destinations never lie above sources.  Every warp counts the flags of a pass for itself.
__device__ __forceinline__ void pack_rows(uint4* kbase, uint4* vbase, const uint8_t* tk, int pb, int pe, int32_t* map) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int r = tid >> 4, col = tid & 15;                // rows r and r + 64 of a pass
    int done = pb;
    for (int cb = pb; cb < pe; cb += 128) {
        unsigned m[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) m[q] = __ballot_sync(0xffffffffu, cb + q * 32 + lane < pe && tk[cb + q * 32 + lane] != 0);
        const int n0 = __popc(m[0]), n1 = n0 + __popc(m[1]), n2 = n1 + __popc(m[2]);
        const unsigned below = (1u << (r & 31)) - 1u;
        const unsigned ma = r < 32 ? m[0] : m[1], mb = r < 32 ? m[2] : m[3];
        const int da = done + (r < 32 ? 0 : n0) + __popc(ma & below), db = done + (r < 32 ? n1 : n2) + __popc(mb & below);
        const int ta = cb + r, tb = ta + 64;
        const bool fa = (ma >> (r & 31)) & 1u, fb = (mb >> (r & 31)) & 1u;
        uint4 k0 = make_uint4(0u, 0u, 0u, 0u), v0 = k0, k1 = k0, v1 = k0;
        if (fa && da != ta) { k0 = kbase[size_t(ta) * 16 + col]; v0 = vbase[size_t(ta) * 16 + col]; }
        if (fb && db != tb) { k1 = kbase[size_t(tb) * 16 + col]; v1 = vbase[size_t(tb) * 16 + col]; }
        if (map && col == 0) {
            if (fa) map[da - pb] = ta;
            if (fb) map[db - pb] = tb;
        }
        done += n2 + __popc(m[3]);
        __syncthreads();
        if (fa && da != ta) { kbase[size_t(da) * 16 + col] = k0; vbase[size_t(da) * 16 + col] = v0; }
        if (fb && db != tb) { kbase[size_t(db) * 16 + col] = k1; vbase[size_t(db) * 16 + col] = v1; }
        __syncthreads();
    }
}

// What the plan leaves for the move, by slab.
struct PlanOut {
    int32_t *len, *nruns, *run_src, *run_dst, *seg_run, *seg_dep;
    uint32_t* loaded;
    int segs;
};

// Bound by latency (one CTA per slab, a few KB each): the table is read together with its length, and partly kept sentences are
// counted by a warp each.
template <bool kFill>
__global__ void __launch_bounds__(kPlanThreads)
compact_plan_kernel(int Hk, int max_sent, const int64_t* slab_off, const int32_t* cap, const uint8_t* keep,
                    const uint8_t* tok_keep, uint4* K, uint4* V, int32_t* sent_off, int32_t* sent_id, int32_t* n_sent,
                    int32_t* kv_len, int32_t* index_map, Header* hdr, PlanOut out) {
    __shared__ int wsum[kPlanThreads / 32][3];
    __shared__ int s_bad, s_total;
    __shared__ int s_npart, s_part[kMaxPartial][3];
    __shared__ int s_nlist, s_list[kFill ? kPlanThreads : 1], s_klen[kFill ? kPlanThreads : 1];
    __shared__ int s_last[kPlanThreads / 32];
    __shared__ int s_next_begin[2];                      // old sent_off[base] of the next chunk of sentences (by chunk parity)
    // the move kernel is launched as a programmatic dependent: let its CTAs set themselves up while this grid runs
    pdl_trigger();
    const int slab = blockIdx.x;
    const int b = slab / Hk;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) { s_npart = 0; s_nlist = 0; s_total = 0; }
    pdl_wait();                                          // inputs may come from the kernel before
    const uint8_t* kp = keep + size_t(slab) * max_sent;
    int32_t* so = sent_off + size_t(slab) * (max_sent + 1);
    int32_t* sid = sent_id + size_t(slab) * max_sent;
    int32_t* run_src = out.run_src + size_t(slab) * max_sent;
    int32_t* run_dst = out.run_dst + size_t(slab) * (max_sent + 1);
    int32_t* seg_run = out.seg_run + size_t(slab) * out.segs;
    int32_t* seg_dep = out.seg_dep + size_t(slab) * out.segs;
    // the first chunk of the table, read along with its length
    int b_i = 0, e_i = 0, id_i = -1, k_i = 0;
    if (tid < max_sent) { b_i = so[tid]; e_i = so[tid + 1]; id_i = sid[tid]; k_i = kp[tid]; }
    const int S = n_sent[slab];
    const int capb = min(cap[b], (out.segs - 1) * kSegRows);
    const size_t row0 = slab_row0(slab_off, cap, Hk, b, slab % Hk);
    const uint8_t* tk = kFill ? tok_keep + row0 : nullptr;
    if (tid == 0) {
        s_bad = (S < 0 || S > max_sent) ? 1 : 0;
        if (slab == 0) hdr->compact_ticket = 0u;
    }
    __syncthreads();
    if (s_bad) {
        if (tid == 0) { atomicOr(&hdr->status, SKIPKV_STATUS_BAD_TABLE); out.len[slab] = 0; out.nruns[slab] = 0; }
        return;
    }
    int c_len = 0, c_cnt = 0, c_run = 0;     // carries: kept tokens, kept sentences, runs so far
    int prev_alive_carry = 0;
    for (int base = 0; base < S; base += kPlanThreads) {
        const int i = base + tid;
        int alive = 0, klen = 0;
        bool counted = false;
        if (i < S) {
            if (base > 0) {
                // the table is rewritten in place, and the chunk before may already have overwritten so[base]: its
                // last thread parked the old value
                b_i = tid == 0 ? s_next_begin[((base / kPlanThreads) & 1) ^ 1] : so[i];
                e_i = so[i + 1]; id_i = sid[i]; k_i = kp[i];
            }
            if (tid == kPlanThreads - 1) s_next_begin[(base / kPlanThreads) & 1] = e_i;   // for thread 0 of the next chunk
            if (i == S - 1) s_total = e_i;
            if (b_i < 0 || e_i < b_i || e_i > capb || (i == 0 && b_i != 0)) atomicOr(&s_bad, 1);
            else if (k_i != 0 && e_i > b_i) {
                klen = e_i - b_i;
                counted = kFill && k_i == 2;             // partly kept: its survivors are counted below
            }
        }
        if (kFill) {
            if (counted) { const int q = atomicAdd(&s_nlist, 1); s_list[q] = tid; s_klen[tid] = b_i; }
            __syncthreads();
            const int nl = s_nlist;
            for (int q = warp; q < nl; q += kPlanThreads / 32) {
                const int who = s_list[q], pb = s_klen[who], pe = so[base + who + 1];
                int n = 0;
                for (int t = pb + lane; t < pe; t += 32) n += tk[t] != 0 ? 1 : 0;
                n = __reduce_add_sync(0xffffffffu, n);
                __syncwarp();
                if (lane == 0) s_klen[who] = n;
            }
            __syncthreads();
            if (tid == 0) s_nlist = 0;
            if (counted) klen = s_klen[tid];
        }
        if (klen > 0) alive = klen < e_i - b_i ? 3 : 1;  // bit 1: rows are missing behind this sentence
        const int partial = alive == 3;
        // does the previous sentence also survive, whole?  (adjacent whole survivors form one run; a partly
        // kept sentence is a run of its own)
        int prev_alive = __shfl_up_sync(0xffffffffu, alive, 1);
        if (lane == 31) s_last[warp] = alive;
        __syncthreads();
        if (lane == 0) prev_alive = (tid == 0) ? prev_alive_carry : s_last[warp - 1];
        const int last_alive = s_last[kPlanThreads / 32 - 1];
        const int start = (alive && (prev_alive != 1 || partial)) ? 1 : 0;
        alive = alive ? 1 : 0;
        int x_len, x_cnt, x_run, tot[3];
        block_scan3(klen, alive, start, x_len, x_cnt, x_run, tot, wsum);   // syncs: old values are all read
        const int dst = c_len + x_len;
        if (alive && !s_bad) {                           // (with a broken table the totals mean nothing)
            so[c_cnt + x_cnt + 1] = dst + klen;
            sid[c_cnt + x_cnt] = id_i;
            const int run = c_run + x_run - (start ? 0 : 1);
            if (start) {
                run_src[run] = partial ? ~b_i : b_i;
                run_dst[run] = dst;
            }
            for (int j = (dst + kSegRows - 1) / kSegRows; j * kSegRows < dst + klen; ++j) seg_run[j] = run;
            if (kFill && partial) {
                const int q = atomicAdd(&s_npart, 1);
                if (q < kMaxPartial) { s_part[q][0] = b_i; s_part[q][1] = e_i; s_part[q][2] = dst; }
                else atomicOr(&s_bad, 1);
            }
        }
        if (i < S && !s_bad)
            for (int j = (b_i + kSegRows - 1) / kSegRows; j * kSegRows < e_i; ++j) seg_dep[j] = dst + min(j * kSegRows - b_i, klen);
        c_len += tot[0]; c_cnt += tot[1]; c_run += tot[2];
        prev_alive_carry = last_alive;
        __syncthreads();
    }
    if (s_bad) {
        // tables may be half rewritten; flag it and move nothing
        if (tid == 0) { atomicOr(&hdr->status, SKIPKV_STATUS_BAD_TABLE); out.len[slab] = 0; out.nruns[slab] = 0; }
        return;
    }
    const int nseg = (c_len + kSegRows - 1) / kSegRows;
    for (int i = c_cnt + 1 + tid; i <= max_sent; i += kPlanThreads) so[i] = c_len;
    for (int i = c_cnt + tid; i < max_sent; i += kPlanThreads) sid[i] = -1;
    uint32_t* loaded = out.loaded + size_t(slab) * 2 * out.segs;
    for (int j = tid; j < nseg; j += kPlanThreads) { loaded[j] = 0u; loaded[out.segs + j] = 0u; }
    if (tid == 0) {
        so[0] = 0;
        run_dst[c_run] = c_len;
        n_sent[slab] = c_cnt;
        kv_len[slab] = c_len;
        out.nruns[slab] = c_run;
        out.len[slab] = c_len;
        for (int j = (s_total + kSegRows - 1) / kSegRows; j <= nseg; ++j) seg_dep[j] = c_len;
    }
    if (kFill) {
        const int np = s_npart;
        for (int q = 0; q < np; ++q)                       // uniform over the CTA
            pack_rows(K + row0 * 16, V + row0 * 16, tk, s_part[q][0], s_part[q][1],
                      index_map ? index_map + row0 + s_part[q][2] : nullptr);
    }
}

__global__ void __launch_bounds__(kMoveThreads)
compact_move_kernel(int n_slabs, int Hk, int max_sent, const int64_t* slab_off, const int32_t* cap,
                    __nv_bfloat16* K, __nv_bfloat16* V, int32_t* index_map, Header* hdr, PlanOut plan,
                    const int32_t* block_table, int max_pages) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int s_red[kMoveThreads / 32];
    __shared__ uint32_t s_ticket[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid == 0) { mbar_init(&bar, 1); mbar_fence_init(); }
    // everything below reads what the plan kernel wrote: wait until that grid has completed and its writes are visible
    pdl_wait();
    pdl_trigger();                                       // every CTA is resident: the next kernel's may set themselves up
    if (tid == 0) s_ticket[0] = atomicAdd(&hdr->compact_ticket, 1u);
    // every CTA derives the scheduler bound: the largest segment count of any slab
    int mx = 0;
    for (int i = tid; i < n_slabs; i += kMoveThreads) mx = max(mx, plan.len[i]);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) s_red[warp] = mx;
    const uint32_t limit = load_wait_limit(hdr);       // polls a wait makes before it gives up
    __syncthreads();
    int max_len = 0;
    for (int w = 0; w < kMoveThreads / 32; ++w) max_len = max(max_len, s_red[w]);
    const uint32_t n_streams = 2u * n_slabs;
    const uint32_t n_tickets = n_streams * uint32_t((max_len + kSegRows - 1) / kSegRows);
    uint32_t phase = 0;

    for (uint32_t it = 0;; ++it) {
        __syncthreads();                               // the ticket is written
        const uint32_t T = s_ticket[it & 1];
        if (T >= n_tickets) break;                     // (the same value for every thread: a uniform exit)
        uint32_t next = 0;
        if (tid == 0) next = atomicAdd(&hdr->compact_ticket, 1u);
        const int stream = int(T % n_streams), j = int(T / n_streams);
        const int slab = stream >> 1;
        const int b = slab / Hk, h = slab % Hk;
        // what the plan knows of this segment: independent loads
        const int new_len = plan.len[slab], nruns = plan.nruns[slab];
        const int r0 = plan.seg_run[size_t(slab) * plan.segs + j];
        const int dep0 = plan.seg_dep[size_t(slab) * plan.segs + j], dep1 = plan.seg_dep[size_t(slab) * plan.segs + j + 1];
        // contiguous slabs: token t of the slab is row row0 + t; paged cache (128-row pages): row table[t / 128] * 128 + t % 128,
        // and a copy is cut where its source or its destination crosses a page
        const int32_t* table = block_table ? block_table + size_t(slab) * max_pages : nullptr;
        const size_t row0 = table ? size_t(slab) * max_pages * 128 : slab_row0(slab_off, cap, Hk, b, h);   // (paged: index_map rows)
        const int d0 = j * kSegRows, d1 = min(d0 + kSegRows, new_len);
        if (d0 >= d1) {                                // a shorter slab
            if (tid == 0) s_ticket[(it + 1) & 1] = next;
            continue;
        }
        uint8_t* tensor = reinterpret_cast<uint8_t*>((stream & 1) ? V : K);
        uint8_t* base = tensor + (table ? 0 : row0 * kRowBytes);
        auto row_ptr = [&](int t) {
            return table ? tensor + (size_t(max(table[t >> 7], 0)) * 128 + (t & 127)) * kRowBytes : base + size_t(t) * kRowBytes;
        };
        auto piece_rows = [&](int src, int dst, int left) {      // rows of a copy that stay inside one page on both sides
            return table ? min(left, min(128 - (src & 127), 128 - (dst & 127))) : left;
        };
        const int32_t* run_src = plan.run_src + size_t(slab) * max_sent;
        const int32_t* run_dst = plan.run_dst + size_t(slab) * (max_sent + 1);
        // destination rows [ps, pe) of run r inside the segment come from token src on; false: the run lies behind it
        auto piece = [&](int r, int& ps, int& pe, int& src, bool& mapped) {
            if (r >= nruns) return false;
            const int rd = run_dst[r], re = run_dst[r + 1], rs = run_src[r];
            if (rd >= d1) return false;
            ps = max(rd, d0); pe = min(re, d1);
            mapped = rs < 0;
            src = (rs < 0 ? ~rs : rs) + (ps - rd);
            return true;
        };
        int ps, pe, src;
        bool mapped;
        if (warp == 0) {
            uint32_t* loaded = plan.loaded + size_t(stream) * plan.segs;
            // pass 1: bytes this segment will receive; pass 2: issue the copies
            uint32_t bytes = 0;
            for (int r = r0 + lane; piece(r, ps, pe, src, mapped); r += 32)
                if (src != ps) bytes += uint32_t(pe - ps) * kRowBytes;
            bytes = __reduce_add_sync(0xffffffffu, bytes);
            if (lane == 0) {
                if (bytes) mbar_expect_tx(&bar, bytes); else mbar_arrive(&bar);
            }
            __syncwarp();
            for (int r = r0 + lane; piece(r, ps, pe, src, mapped); r += 32)
                if (src != ps)
                    for (int o = 0; o < pe - ps;) {
                        const int nr = piece_rows(src + o, ps + o, pe - ps - o);
                        bulk_g2s(smem + size_t(ps + o - d0) * kRowBytes, row_ptr(src + o), uint32_t(nr) * kRowBytes, &bar);
                        o += nr;
                    }
            // the segments whose source rows lie inside this one (a lane each; never more than two, as they hold at most kSegRows survivors)
            const int dep = dep0 / kSegRows + lane;
            const bool has_dep = dep < j && dep * kSegRows < dep1;
            volatile uint32_t* flag = loaded + dep;
            bool open = has_dep && *flag == 0u;
            // every lane observes the landing of the loads it is about to forward
            bool ok = mbar_wait(&bar, phase, limit);
            if (!ok) atomicOr(&hdr->status, SKIPKV_STATUS_COPY_TIMEOUT);
            __syncwarp();
            if (lane == 0) {
                __threadfence();
                *reinterpret_cast<volatile uint32_t*>(loaded + j) = 1u;
            }
            uint32_t spins = 0;
            while (open) {
                if (++spins > limit) {
                    ok = false;
                    atomicOr(&hdr->status, SKIPKV_STATUS_COMPACT_TIMEOUT);
                    break;
                }
                __nanosleep(32);
                open = *flag == 0u;
            }
            __threadfence();
            __syncwarp();                              // what one lane saw comes before every lane's stores
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                for (int r = r0 + lane; piece(r, ps, pe, src, mapped); r += 32)
                    if (src != ps)
                        for (int o = 0; o < pe - ps;) {
                            const int nr = piece_rows(src + o, ps + o, pe - ps - o);
                            bulk_s2g(row_ptr(ps + o), smem + size_t(ps + o - d0) * kRowBytes, uint32_t(nr) * kRowBytes);
                            o += nr;
                        }
                bulk_commit();
            } else {
                // A wait ran out (flagged above): the stores of this segment are skipped and this CTA stops.  Its own
                // loads may still be in flight towards its shared memory, and they must land before it retires.
                mbar_wait(&bar, phase, 1u << 20);
                next = 0xffffffffu;
            }
            bulk_wait_read_all();                      // shared memory may be refilled
            __syncwarp();
            if (lane == 0) s_ticket[(it + 1) & 1] = next;
        } else if (index_map != nullptr && (stream & 1) == 0) {
            // destination token k of a run came from token run_src + (k - run_dst)
            int32_t* im = index_map + row0;
            for (int r = r0; piece(r, ps, pe, src, mapped); ++r)
                if (!mapped)
                    for (int k = ps + lane; k < pe; k += 32) im[k] = k + (src - ps);
        }
        phase ^= 1u;
    }
    if (warp == 0) bulk_wait_all();                    // all stores performed before exit
}

}  // namespace skipkv

using namespace skipkv;

static int compact_impl(const skipkv_shape* shape, void* K, void* V, const uint8_t* keep, const uint8_t* tok_keep,
                        int32_t* sent_off, int32_t* sent_id, int32_t* n_sent, int32_t* kv_len, int32_t* index_map,
                        void* ws, void* stream, const int32_t* block_table = nullptr, int max_pages = 0) {
    if (int rc = check_shape(shape)) return rc;
    if (!K || !V || !keep || !sent_off || !sent_id || !n_sent || !kv_len) return SKIPKV_ERR_INVALID_ARG;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return SKIPKV_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(K) & 15) || (reinterpret_cast<uintptr_t>(V) & 15)) return SKIPKV_ERR_INVALID_ARG;
    const WsLayout L = make_layout(*shape);
    uint8_t* w = static_cast<uint8_t*>(ws);
    Header* hdr = reinterpret_cast<Header*>(w + L.header);
    PlanOut plan;
    plan.len = reinterpret_cast<int32_t*>(w + L.cp_len);
    plan.nruns = reinterpret_cast<int32_t*>(w + L.cp_nruns);
    plan.run_src = reinterpret_cast<int32_t*>(w + L.cp_run_src);
    plan.run_dst = reinterpret_cast<int32_t*>(w + L.cp_run_dst);
    plan.seg_run = reinterpret_cast<int32_t*>(w + L.cp_seg_run);
    plan.seg_dep = reinterpret_cast<int32_t*>(w + L.cp_seg_dep);
    plan.loaded = reinterpret_cast<uint32_t*>(w + L.cp_loaded);
    plan.segs = L.cp_segs;
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    SKIPKV_CUDA(launch_dependent(tok_keep ? compact_plan_kernel<true> : compact_plan_kernel<false>, dim3(L.slabs), dim3(kPlanThreads),
                                 0, st, int(shape->n_kv_heads), int(shape->max_sent), shape->slab_off, shape->cap, keep, tok_keep,
                                 static_cast<uint4*>(K), static_cast<uint4*>(V), sent_off, sent_id, n_sent, kv_len, index_map, hdr,
                                 plan));
    SKIPKV_CUDA(launch_dependent(compact_move_kernel, dim3(unsigned(num_sms() * kMoveCtas)), dim3(kMoveThreads), kSegBytes, st,
                                 int(L.slabs), int(shape->n_kv_heads), int(shape->max_sent), shape->slab_off, shape->cap,
                                 static_cast<__nv_bfloat16*>(K), static_cast<__nv_bfloat16*>(V), index_map, hdr, plan, block_table,
                                 max_pages));
    return SKIPKV_OK;
}

extern "C" int skipkv_compact(const skipkv_shape* shape, void* K, void* V, const uint8_t* keep,
                              int32_t* sent_off, int32_t* sent_id, int32_t* n_sent, int32_t* kv_len,
                              int32_t* index_map, void* ws, void* stream) {
    return compact_impl(shape, K, V, keep, nullptr, sent_off, sent_id, n_sent, kv_len, index_map, ws, stream);
}

extern "C" int skipkv_compact_fill(const skipkv_shape* shape, void* K, void* V, const uint8_t* keep,
                                   const uint8_t* tok_keep, int32_t* sent_off, int32_t* sent_id, int32_t* n_sent,
                                   int32_t* kv_len, int32_t* index_map, void* ws, void* stream) {
    if (!tok_keep) return SKIPKV_ERR_INVALID_ARG;
    return compact_impl(shape, K, V, keep, tok_keep, sent_off, sent_id, n_sent, kv_len, index_map, ws, stream);
}

extern "C" int skipkv_compact_paged(const skipkv_shape* shape, void* K_pages, void* V_pages, const int32_t* block_table,
                                    int32_t max_pages, const uint8_t* keep, int32_t* sent_off, int32_t* sent_id,
                                    int32_t* n_sent, int32_t* kv_len, int32_t* index_map, void* ws, void* stream) {
    if (!block_table || max_pages <= 0) return SKIPKV_ERR_INVALID_ARG;
    return compact_impl(shape, K_pages, V_pages, keep, nullptr, sent_off, sent_id, n_sent, kv_len, index_map, ws, stream,
                        block_table, max_pages);
}
