// skipkv_token_redundancy: the token-redundancy term at TOKEN granularity (paper Section 4.1,
// token-redundancy equation: R = mean(softmax(Kbar Kbar^T)) with Kbar = K / (||K||_2 + eps)), an
// N' x N' Gram matrix per (sequence, KV head) slab over the slab's own key rows:
//     G_ij  = K_i . K_j / ((|K_i| + eps)(|K_j| + eps))
//     Z_j   = sum_{k != j} exp(G_jk)
//     R_i   = (1/N') sum_{j != i} exp(G_ji) / Z_j
// Four launches:
//   token_norm_kernel      1 / (|K_t| + eps) of every live row (a warp per row); clears Z and R;
//   token_red_kernel<1>    row sums Z;
//   token_red_kernel<2>    R, without the 1/N' and less its mean;
//   token_mean_kernel      both.
// G is symmetric, so every pair of 128-row blocks {I, J} is multiplied and exponentiated once: the tile gives the
// rows of I their sums over the columns and the rows of J theirs as column sums.  A work item is block J of a slab as
// columns against itself and the blocks after it as rows, cyclically, half-way round: every pair once, all items of a
// slab equally long.  Z and R are accumulated with floating-point reductions: sums agree to rounding, not to the bit,
// from run to run.  A value of R gets about N/64 contributions, each of which would be rounded at the magnitude of the sum; so every
// contribution comes less tr_mean(N), about 1/N, for each of its terms, what is accumulated stays small, and token_mean_kernel
// adds what was left out: error against 64 bits 8.6e-8 -> 2.3e-8 at 4224 rows, 1.27e-7 -> 3.5e-8 at 7611 (one reduction after the other
// from zero; with half as many of them it had been 5.8e-8 and 9.0e-8), for 617 -> 628 us (80 slabs x 4224 rows).
// The Gram kernels are persistent and warp-specialised.  Warp 0 streams the bf16 key tiles straight from the cache
// with tiled TMA loads (the J tile once per item, the I tiles through a ring), warps 1 and 2 issue one
// 128 x 128 x 128 tcgen05.mma group per block pair in turn into one of four tensor-memory accumulators (a single issuer
// leaves the tensor pipe idle while it waits on its barriers), and sixteen warps read every accumulator back, 32
// rows x 32 columns each, scale by the two inverse norms and exponentiate.  The products of bf16 keys are exact in fp32,
// so no operand is rounded: normalisation happens after the contraction.
// The columns of an item stay the same from tile to tile, so a thread keeps its 32 column sums in registers and the lanes are added
// up once per item; with the rows fixed and the columns streamed, that butterfly (31 exchanges and as many selects for 32
// elements) came with every tile and took longer than the exponentials.
// What bounds it: the epilogue, none of whose units is saturated: the schedulers issue on 6 clocks of 10, exponentials (8 clocks of a
// scheduler for a warp) take 61 to 65 % of their unit, the tensor pipe is at 29 to 32 %.  A warp waits for an accumulator, loads it and works
// on it in sequence; four warps per scheduler hide most of that, two with 64 columns each do not (326 us a pass).  A share of the
// exponentials as polynomials took 10 % more.  80 slabs x 4224 keys, both passes and the norms: 804 -> 617 us
// back to back (558 in a short burst: the clock falls under the power limit), before the mean was kept apart.
#include "tc.cuh"

namespace skipkv {

constexpr int kTrAcc = 4;                    // tensor-memory accumulators of 128 columns
constexpr int kTrThreads = 20 * 32;          // TMA warp, two MMA warps, one idle, four epilogue warpgroups
constexpr int kTrStages = 4;                 // row tiles in flight
constexpr float kTrLog2e = 1.4426950408889634f;

struct TrCtl {
    uint64_t jfull[2], jempty[2], ifull[kTrStages], iempty[kTrStages], tfull[kTrAcc], tempty[kTrAcc];
    uint32_t tmem_base;
    int abort_flag;
    uint32_t wsum[32];
    alignas(16) float col[16][2][32];        // by epilogue warp: log2(e) / (|K_j| + eps) of its columns; pass 2: 1 / Z_j
    uint64_t retired[2];                     // every product of an MMA warp has completed
};
constexpr size_t kTrSmem = 1024 + (2 + kTrStages) * size_t(kOpBytes) + sizeof(TrCtl);          // and the table of slabs behind it

// Blocks that item (slab of NB blocks, block J) multiplies block J with: J itself and the next ones, cyclically.
__device__ __forceinline__ int tr_count(int NB, int I) {
    const int half = NB >> 1;
    return (NB & 1) ? 1 + half : half + (I < half ? 1 : 0);
}
// 1/N to 12 bits, so that a few thousand times it is exact.
__device__ __forceinline__ float tr_mean(int N) { return __uint_as_float(__float_as_uint(1.f / float(max(N, 1))) & 0xfffff000u); }
__device__ __forceinline__ float tr_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__global__ void __launch_bounds__(256)
token_norm_kernel(int Hk, int max_cap, const int64_t* slab_off, const int32_t* cap, const __nv_bfloat16* K,
                  const int32_t* kv_len, float eps, float* inv_norm, float* z, float* tok_red) {
    const int slab = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_trigger();
    pdl_wait();
    const int len = min(max(kv_len[slab], 0), min(cap[slab / Hk], max_cap));
    const int t0 = blockIdx.x * 64 + warp * 8;
    if (t0 >= len) return;
    const size_t row0 = slab_row0(slab_off, cap, Hk, slab / Hk, slab % Hk);
    uint2 x[8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
        x[r] = (t0 + r < len) ? reinterpret_cast<const uint2*>(K + (row0 + t0 + r) * kHeadDim)[lane] : make_uint2(0u, 0u);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const float a = bf16lo(x[r].x), b = bf16hi(x[r].x), c = bf16lo(x[r].y), d = bf16hi(x[r].y);
        float ss = a * a + b * b + c * c + d * d;
#pragma unroll
        for (int s = 16; s; s >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, s);
        if (lane == 0 && t0 + r < len) {
            inv_norm[size_t(slab) * max_cap + t0 + r] = 1.f / (sqrtf(ss) + eps);
            z[size_t(slab) * max_cap + t0 + r] = 0.f;            // both are accumulated by the passes that follow
            tok_red[row0 + t0 + r] = 0.f;
        }
    }
}

struct TrItem { int slab, S, NB, J, NJ; size_t sbase; };

// Table of slabs in global memory, for calls with more slabs than shared memory has room for beside the tiles.
__global__ void __launch_bounds__(1024)
token_table_kernel(int n_slabs, int Hk, int max_cap, const int32_t* cap, const int32_t* kv_len, int* table) {
    __shared__ uint32_t wsum[32];
    pdl_trigger();
    pdl_wait();
    cta_prefix<1024>(n_slabs, [&](int s) { return (min(max(kv_len[s], 0), min(cap[s / Hk], max_cap)) + 127) >> 7; }, table, wsum);
}

// kTable: the table of slabs is in global memory (an instance of its own: the other one keeps its accesses to shared memory)
template <int kPass, bool kTable>
__global__ void __launch_bounds__(kTrThreads, 1)
token_red_kernel(const __grid_constant__ CUtensorMap mapK, int n_slabs, int Hk, int max_cap, const int64_t* slab_off,
                 const int32_t* cap, const int32_t* kv_len, const float* inv_norm, float* z, float* tok_red,
                 const Header* hdr, int* table) {
    extern __shared__ uint8_t tr_smem_raw[];
    const uint32_t raw = smem_u32(tr_smem_raw);
    uint8_t* Jt = tr_smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint8_t* It = Jt + 2 * kOpBytes;
    TrCtl* ctl = reinterpret_cast<TrCtl*>(It + kTrStages * kOpBytes);
    int* ipref = kTable ? table : reinterpret_cast<int*>(ctl + 1);               // [n_slabs + 1] prefix of blocks
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, cta = blockIdx.x;
    auto len_of = [&](int s) { return min(max(kv_len[s], 0), min(cap[s / Hk], max_cap)); };
    pdl_trigger();

    if (tid == 0) {
        for (int s = 0; s < 2; ++s) { mbar_init(&ctl->jfull[s], 1); mbar_init(&ctl->jempty[s], 2); mbar_init(&ctl->retired[s], 1); }
        for (int s = 0; s < kTrStages; ++s) { mbar_init(&ctl->ifull[s], 1); mbar_init(&ctl->iempty[s], 1); }
        for (int s = 0; s < kTrAcc; ++s) { mbar_init(&ctl->tfull[s], 1); mbar_init(&ctl->tempty[s], 16); }
        ctl->abort_flag = 0;
        mbar_fence_init();
        tmap_prefetch(&mapK);
    }
    if (warp == 1) tmem_alloc(&ctl->tmem_base, 128 * kTrAcc);
    pdl_wait();                                          // kv_len and the norms may come from the kernels before
    uint32_t* status = const_cast<uint32_t*>(&hdr->status);
    const uint32_t limit = load_wait_limit(hdr);
    tc_fence_before();
    if (kTable) __syncthreads();
    else cta_prefix<kTrThreads>(n_slabs, [&](int s) { return (len_of(s) + 127) >> 7; }, ipref, ctl->wsum);   // blocks per slab
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const int n_items = ipref[n_slabs];
    auto row0_of = [&](int s) { return int(slab_row0(slab_off, cap, Hk, s / Hk, s % Hk)); };
    auto get_item = [&](int item, int slab) {            // slab: where to look from
        TrItem x;
        while (ipref[slab + 1] <= item) ++slab;
        x.slab = slab;
        x.S = len_of(slab);
        x.NB = (x.S + 127) >> 7;
        x.J = item - ipref[slab];
        x.NJ = tr_count(x.NB, x.J);
        x.sbase = size_t(slab) * max_cap;
        return x;
    };

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == 0 && lane == 0) {
            bool ok = true;
            int slab = 0;
            uint32_t bc = 0, ic = 0;                                // tiles and items issued so far
            for (int item = cta; item < n_items && ok; item += G, ++ic) {
                const TrItem x = get_item(item, slab);
                slab = x.slab;
                const int row0 = row0_of(slab), js = ic & 1;
                if (ic >= 2) ok = role_wait(&ctl->jempty[js], ((ic >> 1) - 1) & 1u, limit, &ctl->abort_flag, status);
                if (!ok) break;
                mbar_expect_tx(&ctl->jfull[js], kOpBytes);
                tma_load_2d(Jt + js * kOpBytes, &mapK, 0, row0 + x.J * 128, &ctl->jfull[js]);
                tma_load_2d(Jt + js * kOpBytes + kOpHalfBytes, &mapK, 64, row0 + x.J * 128, &ctl->jfull[js]);
                int I = x.J;
                for (int t = 0; t < x.NJ && ok; ++t, ++bc) {
                    const int s = bc % kTrStages;
                    if (bc >= kTrStages) ok = role_wait(&ctl->iempty[s], ((bc / kTrStages) - 1) & 1u, limit, &ctl->abort_flag, status);
                    if (!ok) break;
                    uint8_t* dst = It + size_t(s) * kOpBytes;
                    mbar_expect_tx(&ctl->ifull[s], kOpBytes);
                    tma_load_2d(dst, &mapK, 0, row0 + I * 128, &ctl->ifull[s]);
                    tma_load_2d(dst + kOpHalfBytes, &mapK, 64, row0 + I * 128, &ctl->ifull[s]);
                    if (++I == x.NB) I = 0;
                }
            }
            // Whoever gave up: this warp stays until its copies have landed and the issuers' products have completed, so that the CTA gives
            // back shared and tensor memory with nothing in flight.
            for (uint32_t s = 0; s < 2; ++s)
                if (ic > s) mbar_wait(&ctl->jfull[s], ((ic - 1 - s) >> 1) & 1u, kRetirePolls);
            for (uint32_t s = 0; s < kTrStages; ++s)
                if (bc > s) mbar_wait(&ctl->ifull[s], ((bc - 1 - s) / kTrStages) & 1u, kRetirePolls);
            for (int s = 0; s < 2; ++s) mbar_wait(&ctl->retired[s], 0u, kRetirePolls);
        } else if ((warp == 1 || warp == 2) && lane == 0) {
            // Two issuers, a tile each in turn (stages and accumulators are four: each is always the same issuer's).  One lane of each runs the loop: the
            // epilogue is what bounds this kernel, and with whole warps here, whose products are issued four times as fast, it took 581 us
            // instead of 572 (80 slabs x 4224 keys).
            const uint32_t me = warp - 1, leader = 1u;
            bool ok = true;
            int slab = 0;
            uint32_t bc = 0, ic = 0;
            for (int item = cta; item < n_items && ok; item += G, ++ic) {
                const TrItem x = get_item(item, slab);
                slab = x.slab;
                ok = role_wait(&ctl->jfull[ic & 1], (ic >> 1) & 1u, limit, &ctl->abort_flag, status);
                const uint32_t jt = smem_u32(Jt + (ic & 1) * kOpBytes);
                for (int t = 0; t < x.NJ && ok; ++t, ++bc) {
                    if ((bc & 1u) != me) continue;
                    const int st = bc % kTrStages, s = bc % kTrAcc;
                    ok = role_wait(&ctl->ifull[st], (bc / kTrStages) & 1u, limit, &ctl->abort_flag, status);
                    if (ok && bc >= kTrAcc) ok = role_wait(&ctl->tempty[s], ((bc / kTrAcc) - 1) & 1u, limit, &ctl->abort_flag, status);
                    if (!ok) break;
                    tc_fence_after();
                    umma_tile_128x128x128(tmem_base + s * 128, smem_u32(It + size_t(st) * kOpBytes), jt, false, leader);
                    umma_commit(&ctl->tfull[s], leader);
                    umma_commit(&ctl->iempty[st], leader);
                }
                if (ok) umma_commit(&ctl->jempty[ic & 1], leader);           // every product of this issuer that reads the column tile has completed
            }
            umma_commit(&ctl->retired[me], leader);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        const int quarter = warp & 3, c0 = ((warp - 4) >> 2) * 32;   // this warp's rows (32 * quarter + lane) and columns
        const uint32_t lane_addr = tmem_base + (uint32_t(quarter * 32) << 16) + c0;
        float* col_s = ctl->col[warp - 4][0];
        const float4* col = reinterpret_cast<const float4*>(col_s);  // two pairs of columns per load
        const float4* colz = col + 8;
        uint32_t acc = 0, parity = 0;
        const uint32_t tfull0 = smem_u32(ctl->tfull);        // tempty lies kTrAcc words behind
        float2 cs[16];
        bool ok = true;
        TrItem x = {};
        int slab = 0;
#pragma unroll 1
        for (int item = cta; item < n_items && ok; item += G) {
            x = get_item(item, slab);
            slab = x.slab;
            const float *inv_p = inv_norm + x.sbase, *z_p = z + x.sbase;
            const int S = x.S, wrap = x.NB * 128, j0 = x.J * 128 + c0;
            float inv_n = 1.f, z_n = 0.f, cn = 1.f, cz = 0.f;
            auto fetch_row = [&](int i) {                    // the row scale of a tile, a tile ahead
                inv_n = 1.f; z_n = 0.f;
                if (i < S) {
                    inv_n = inv_p[i];
                    if (kPass == 2) z_n = z_p[i];
                }
            };
            int i = x.J * 128 + quarter * 32 + lane;
            if (j0 + lane < S) {
                cn = inv_p[j0 + lane];
                if (kPass == 2) cz = z_p[j0 + lane];
            }
            fetch_row(i);
            __syncwarp();
            col_s[lane] = cn * kTrLog2e;
            if (kPass == 2) col_s[32 + lane] = cz > 0.f ? 1.f / cz : 0.f;
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 16; ++k) cs[k] = make_float2(0.f, 0.f);
            const float row_mean = kPass == 2 ? float(min(max(S - j0, 0), 32)) * tr_mean(S) : 0.f;   // of this warp's columns
            float* dst = kPass == 1 ? z + x.sbase : tok_red + row0_of(slab);
            // rows from here on are not all the slab's; where the columns are not, none are good enough for the short path
            const int whole = (x.J + 1) * 128 <= S ? S - 31 + lane : 0;
#pragma unroll 1
            for (int t = 0; t < x.NJ; ++t) {
                const float inv_i = inv_n;
                const float invz_i = (kPass == 2 && z_n > 0.f) ? 1.f / z_n : 0.f;   // the weight of this row in column sums
                int i_next = i + 128;
                if (i_next >= wrap) i_next -= wrap;
                fetch_row(i_next);
                const uint32_t tfull = tfull0 + acc * 8;
                {
                    // (inline: a call would spill the sums)
                    bool r = mbar_try_wait(tfull, parity);
                    for (uint32_t n = 0; !r && n < limit; ++n) {
                        if ((n & 63) == 63 && *reinterpret_cast<volatile int*>(&ctl->abort_flag)) break;
                        r = mbar_try_wait(tfull, parity);
                    }
                    ok = __all_sync(0xffffffffu, r);
                    tc_fence_after();
                }
                if (!ok) {
                    atomicOr(status, SKIPKV_STATUS_COPY_TIMEOUT);
                    *reinterpret_cast<volatile int*>(&ctl->abort_flag) = 1;
                    break;
                }
                float2 row = make_float2(-row_mean, 0.f);
                float v[32];
                tmem_ld32(lane_addr + acc * 128, v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tfull + kTrAcc * 8);
                // two elements per instruction (packed fp32 multiply / add)
                const float2 inv2 = make_float2(inv_i, inv_i), iz2 = make_float2(invz_i, invz_i);
                auto scaled = [&](int k, float x0, float x1) { return __fmul2_rn(__fmul2_rn(make_float2(v[2 * k], v[2 * k + 1]), inv2), make_float2(x0, x1)); };
                auto add = [&](int k, float2 e, float z0, float z1) {
                    if (kPass == 1) {
                        row = __fadd2_rn(row, e);
                        cs[k] = __fadd2_rn(cs[k], e);
                    } else {
                        row = __ffma2_rn(e, make_float2(z0, z1), row);
                        cs[k] = __ffma2_rn(e, iz2, cs[k]);
                    }
                };
                if (t > 0 && i < whole) {                    // (the same for the whole warp)
#pragma unroll
                    for (int k = 0; k < 16; k += 2) {
                        const float4 c = col[k / 2], cz4 = kPass == 2 ? colz[k / 2] : c;
                        const float2 w = scaled(k, c.x, c.y), u = scaled(k + 1, c.z, c.w);
                        add(k, make_float2(tr_ex2(w.x), tr_ex2(w.y)), cz4.x, cz4.y);
                        add(k + 1, make_float2(tr_ex2(u.x), tr_ex2(u.y)), cz4.z, cz4.w);
                    }
                } else {                                     // nothing where a row or column is none of the slab's, and for i == j
                    const int lim = i < S ? S - j0 : 0, self = i - j0;
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const float2 c = reinterpret_cast<const float2*>(col)[k], cz2 = kPass == 2 ? reinterpret_cast<const float2*>(colz)[k] : c;
                        const float2 w = scaled(k, c.x, c.y);
                        add(k, make_float2(2 * k < lim && 2 * k != self ? tr_ex2(w.x) : 0.f,
                                           2 * k + 1 < lim && 2 * k + 1 != self ? tr_ex2(w.y) : 0.f), cz2.x, cz2.y);
                    }
                }
                // (the block against itself is symmetric: its column sums are all there is to it)
                if (t > 0 && i < S) atomicAdd(dst + i, row.x + row.y);
                i = i_next;
                if (++acc == kTrAcc) { acc = 0; parity ^= 1u; }
            }
            if (ok) {
                // the same exponentials as column sums: they belong to the rows of block J
                float s[32];
#pragma unroll
                for (int k = 0; k < 16; ++k) { s[2 * k] = cs[k].x; s[2 * k + 1] = cs[k].y; }
                float sum = col_reduce32(s, lane);
                if (kPass == 2) {                            // this warp's rows in the item's blocks, the last of which may be partly filled, less the token itself
                    const int short_of = x.J + x.NJ >= x.NB ? 32 - min(max(x.S - (x.NB - 1) * 128 - quarter * 32, 0), 32) : 0;
                    sum -= float(32 * x.NJ - short_of - (quarter * 32 == c0 ? 1 : 0)) * tr_mean(x.S);
                }
                if (j0 + lane < x.S) atomicAdd(dst + j0 + lane, sum);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 128 * kTrAcc);
    }
}

__global__ void __launch_bounds__(256)
token_mean_kernel(int Hk, int max_cap, const int64_t* slab_off, const int32_t* cap, const int32_t* kv_len, float* tok_red) {
    pdl_trigger();
    pdl_wait();
    const int slab = blockIdx.y, t0 = blockIdx.x * 1024 + threadIdx.x;
    const int len = min(max(kv_len[slab], 0), min(cap[slab / Hk], max_cap));
    float* dst = tok_red + slab_row0(slab_off, cap, Hk, slab / Hk, slab % Hk);
    if (len == 0) return;
    const double rest = double(len - 1) * double(tr_mean(len)), inv = 1.0 / double(len);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (t0 + k * 256 < len) dst[t0 + k * 256] = float((double(dst[t0 + k * 256]) + rest) * inv);
}

}  // namespace skipkv

using namespace skipkv;

extern "C" int skipkv_token_redundancy(const skipkv_shape* shape, const skipkv_params* params, const void* K,
                                       const int32_t* kv_len, float* tok_red, void* ws, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!params || !K || !kv_len || !tok_red) return SKIPKV_ERR_INVALID_ARG;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return SKIPKV_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(K) & 15) return SKIPKV_ERR_INVALID_ARG;
    const WsLayout L = make_layout(*shape);
    uint8_t* w = static_cast<uint8_t*>(ws);
    const Header* hdr = reinterpret_cast<const Header*>(w + L.header);
    float* inv_norm = reinterpret_cast<float*>(w + L.tr_inv);
    float* z = reinterpret_cast<float*>(w + L.tr_z);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    CUtensorMap mapK;
    if (int rc = tmap_rows(&mapK, K, uint64_t(shape->total_rows), 128)) return rc;
    // The table (4 bytes a slab) goes into shared memory up to about 7600 slabs, the room beside six tiles; beyond that into the workspace.
    size_t smem = kTrSmem + size_t(L.slabs + 1) * 4;
    const bool in_global = smem > 227 * 1024;
    if (in_global) smem = kTrSmem;
    int* table = in_global ? reinterpret_cast<int*>(w + L.slab_table) : nullptr;
    const int Hk = shape->n_kv_heads;
    SKIPKV_CUDA(launch_dependent(token_norm_kernel, dim3((shape->max_cap + 63) / 64, L.slabs), dim3(256), 0, st, Hk,
                                 int(shape->max_cap), shape->slab_off, shape->cap, static_cast<const __nv_bfloat16*>(K),
                                 kv_len, params->eps, inv_norm, z, tok_red));
    const long long max_items = (long long)L.slabs * ((shape->max_cap + 127) / 128);
    int grid = num_sms();
    if (max_items < grid) grid = int(max_items);
    if (in_global)
        SKIPKV_CUDA(launch_dependent(token_table_kernel, dim3(1), dim3(1024), 0, st, int(L.slabs), Hk, int(shape->max_cap), shape->cap,
                                     kv_len, table));
    for (int pass = 1; pass <= 2; ++pass) {
        const auto kernel = pass == 1 ? (in_global ? token_red_kernel<1, true> : token_red_kernel<1, false>)
                                      : (in_global ? token_red_kernel<2, true> : token_red_kernel<2, false>);
        SKIPKV_CUDA(launch_dependent(kernel, dim3(grid), dim3(kTrThreads), smem, st, mapK, int(L.slabs), Hk, int(shape->max_cap),
                                     shape->slab_off, shape->cap, kv_len, static_cast<const float*>(inv_norm), z, tok_red, hdr, table));
    }
    SKIPKV_CUDA(launch_dependent(token_mean_kernel, dim3((shape->max_cap + 1023) / 1024, L.slabs), dim3(256), 0, st, Hk, int(shape->max_cap),
                                 shape->slab_off, shape->cap, kv_len, tok_red));
    return SKIPKV_OK;
}
