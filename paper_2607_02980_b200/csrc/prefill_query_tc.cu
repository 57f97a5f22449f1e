// Query-major prefill on tcgen05 tensor cores (bf16, d = 128, S = 64, G = 4, one landmark per KV head) for the tokens
// that see few chunks.
//
// (And, for the other tokens, the chunks of wide local windows, which neighbours share too: prefill_local_query.)
//
// Where the candidates of a token are not many more than top_k, neighbouring tokens attend mostly the same chunks: a tile of
// 32 tokens x 4 heads (128 MMA rows) walks the union of its tokens' chunks, and the mix of Eq. (HiLS weights) stays in
// tensor memory until `out` is written once.  The chunk-major kernels (prefill_attend_tc.cu) move a query row in and a
// partial output row out and in again per (token, chunk) pair; here a chunk costs a tile one score and one value product,
// whoever of its tokens selected it (the others meet probabilities of zero).
//
// A CTA works on units of 64 adjacent tokens of one (sequence, KV head): two tiles that share the K / V stream, each with
// its own scores, probabilities and output accumulator in tensor memory (256 columns).
//   warps 0-3, 4-7   softmax of tile 0 / 1 (warp = head, lane = token): the chunk's own softmax, its mixing logit (the
//                    landmark is key 64 of the score tile; the exact log mass for a chunk of the local window), normalised
//                    probabilities times the mixing weight as bf16 into tensor memory.  The weights refer to a running
//                    reference logit per row that is raised, and the accumulator scaled, only when a logit exceeds it by
//                    kRaise: rare, and bf16 / fp32 keep their relative precision in between.  At the end of a unit the same
//                    warps write the tile's rows.
//   warps 8, 9       issue the MMAs of tile 0 / 1 (the next chunk's scores before this chunk's value product)
//   warp 10          loads K, V, landmark rows and queries by TMA
//   warp 11          builds the unit's list of chunks (and which tile needs them, with a bit per token), one unit ahead
// Bound: the softmax warps' serial chain per chunk, 2000 cycles: answer of the barrier 290, tensor-memory load 100, maximum 200, exponentials
// 750 (two warps per scheduler; special-function unit 37 % busy), weight 200, accumulator's answer 170, probabilities back 190.  The
// tensor pipe needs 1350 of them.  The rounded division of w by z took 300 cycles of the chain: 2 x 6000 tokens, K = 32, us for the call with
// it 739, with quotient() 694 (with the approximate quotient, which loses two bits, 686); the next item's barrier is asked early.
// A unit's fixed part: 9300 -> 5000 cycles with the output staged beside the query tile, so that the next unit's queries come with this
// one's last scores, and the unit's place worked out once, by the list warp (this kernel on 2 x 6000 tokens 587 -> 571 us, the call on 3 x 1000 44.9 -> 42.0).
// Sixteen softmax warps, half a row's keys or every other item each: 704 and 781 us (more instructions, colder instruction cache).
#include "internal.h"
#include "tma.cuh"

namespace hils {
namespace {

constexpr int kD = 128;
constexpr int kS = 64;
constexpr int kG = 4;
constexpr int kTok = 32;                        // tokens per tile
constexpr int kUnitTok = 64;                    // tokens per unit
constexpr int kRows = kTok * kG;
constexpr int kNS = 80;                         // score columns: 64 keys + landmark (+ 15 zero rows)
constexpr int kKBytes = kNS * kD * 2;
constexpr int kVBytes = kS * kD * 2;
constexpr int kQBytes = kRows * kD * 2;
constexpr int kStages = 3;
constexpr int kStgBytes = kTok * 128;           // staging of a softmax warp's output: its 32 rows x 64 dimensions
constexpr int kMaxK = 64;                       // selected chunks per token
constexpr int kMaxC = 256;                      // chunks a unit may see
constexpr int kPCol = 96;                       // columns of a tile: scores 0..79, probabilities 96..127, output 128..255
constexpr int kOCol = 128;
constexpr int kMmaWarp = 8, kLoadWarp = 10;           // (and warp 11, the list)
constexpr int kThreads = 12 * 32;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRaise = 16.f;

struct QmArgs {
    Shape s;
    const __nv_bfloat16* lm;
    const float* bias;
    int32_t* sel;
    __nv_bfloat16* out;
    float* lse;
    int* status;
    int first, n_tok;  // tokens first .. n_tok - 1 of every sequence (first: a multiple of 64)
    int local;         // 1: the chunks of the local windows alone; out and lse are then that branch's output and log mass
    int write_sel;     // 1: no token has more candidates than top_k, the selection is written here
};

struct QmSmem {
    uint64_t kv_full[kStages], kv_empty[kStages];
    uint64_t q_full[2], q_empty[2];
    uint64_t s_full[2], s_empty[2], p_full[2], o_done[2];
    uint64_t list_full[2], list_empty[2], ids_full;
    alignas(16) int32_t ids[kMaxK * kTok];      // (list builder) selections of 64 tokens (of 32, more than 32 chunks each)
    uint32_t tmem_base;
    int blk[2], pair[2], seq[2];                // [list] the unit: its block of tokens, (sequence, KV head), sequence
    int n_items[2];                             // items of the unit's list
    int base[2];                                // first chunk of the unit (lists and masks count from it)
    int list[2][kMaxC];                         // chunk | tile 0 needs it << 16 | tile 1 needs it << 17
    uint32_t mask[2][kMaxC];                    // (list builder) [tile][chunk]: tokens that attend it
    int n_tile[2][2];                           // [list][tile]: items of the tile
    int2 titem[2][2][kMaxC];                    // [list][tile][item]: chunk, tokens that attend it
};
static_assert(kStages * (kKBytes + kVBytes) + 2 * kQBytes + kMmaWarp * kStgBytes + sizeof(QmSmem) + 1024 <= 232448, "shared memory of the query-major kernel");

// bit x of a word (none for x < 0 and x > 31)
__device__ __forceinline__ uint32_t bit_or_none(int x) {
    uint32_t r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(x));                       // (the count is unsigned and saturates at 32)
    return r;
}
// the lowest n bits (n < 0: none, n > 31: all)
__device__ __forceinline__ uint32_t bits_below(int n) { return bit_or_none(max(n, 0)) - 1u; }

// 2^x of two values on the FMA pipes: x = n + f with f in [-1/2, 1/2] (Cody-Waite), a polynomial of degree 5 in f fitted
// to the smallest relative error (1e-7), n added to the exponent.  A quarter of a row's exponentials goes this way: the
// special-function unit takes 8 cycles per warp and exponential and is the busiest unit of the softmax warps.
__device__ __forceinline__ float2 ex2_fma(float2 x) {
    x.x = fmaxf(x.x, -126.f);
    x.y = fmaxf(x.y, -126.f);
    const float2 t = __fadd2_rn(x, make_float2(12582912.f, 12582912.f));            // 1.5 * 2^23: rounds to an integer
    const float2 n = __fadd2_rn(t, make_float2(-12582912.f, -12582912.f));
    const float2 f = __ffma2_rn(n, make_float2(-1.f, -1.f), x);
    float2 p = __ffma2_rn(make_float2(0.00132765f, 0.00132765f), f, make_float2(0.00967554f, 0.00967554f));
    p = __ffma2_rn(p, f, make_float2(0.05550713f, 0.05550713f));
    p = __ffma2_rn(p, f, make_float2(0.24022120f, 0.24022120f));
    p = __ffma2_rn(p, f, make_float2(0.69314697f, 0.69314697f));
    p = __ffma2_rn(p, f, make_float2(1.00000007f, 1.00000007f));
    return make_float2(__int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23)),
                       __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23)));
}

__global__ void __launch_bounds__(kThreads, 1)
prefill_query_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                        const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_out, const QmArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* kbuf = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* vbuf = kbuf + kStages * kKBytes;
    uint8_t* qbuf = vbuf + kStages * kVBytes;
    uint8_t* stage = qbuf + 2 * kQBytes;
    QmSmem& sm = *reinterpret_cast<QmSmem*>(stage + kMmaWarp * kStgBytes);
    const Shape& s = a.s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pairs = s.B * s.Hkv, blk0 = a.first / kUnitTok, n_blk = (a.n_tok - a.first + kUnitTok - 1) / kUnitTok, n_units = pairs * n_blk;

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&sm.kv_full[i], 1); mbar_init(&sm.kv_empty[i], 2); }
        for (int t = 0; t < 2; ++t) {
            mbar_init(&sm.q_full[t], 1); mbar_init(&sm.q_empty[t], 1);
            mbar_init(&sm.s_full[t], 1); mbar_init(&sm.s_empty[t], 4);
            mbar_init(&sm.p_full[t], 4); mbar_init(&sm.o_done[t], 1);
            mbar_init(&sm.list_full[t], 1); mbar_init(&sm.list_empty[t], 11);
        }
        mbar_init(&sm.ids_full, 1);
        mbar_fence_init();
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
        tma_prefetch_desc(&map_out);
    }
    // rows 64 .. 79 of every K buffer: the landmark row and zeros (TMA writes rows 0 .. 63)
    for (int x = tid; x < kStages * 2 * 16 * 8; x += kThreads) {
        const int st = x >> 8, kb = (x >> 7) & 1, row = 64 + ((x >> 3) & 15), pc = x & 7;
        *reinterpret_cast<uint4*>(kbuf + st * kKBytes + kb * (kNS * 128) + swz128(row, pc)) = make_uint4(0u, 0u, 0u, 0u);
    }
    if (warp == kMmaWarp) tmem_alloc(&sm.tmem_base, 512);
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = sm.tmem_base;
    pdl_wait();                                  // the selection

    // unit idx: (block of 64 tokens, pair), the blocks with the most chunks first; ln: its list buffer
    // (every other round of the walk runs backwards: the units get lighter along it, and a CTA that was early in one round
    // is late in the next)
    auto unit_of = [&](int idx, int& blk, int& pair) {
        const int rnd = idx / static_cast<int>(gridDim.x);
        if (rnd & 1) {
            const int end = min(n_units, (rnd + 1) * static_cast<int>(gridDim.x)) - 1;
            idx = end - (idx - rnd * static_cast<int>(gridDim.x));
        }
        blk = blk0 + n_blk - 1 - idx / pairs;
        pair = idx % pairs;
    };
    bool ok = true;
    // (a test first: where the phase is over, as it mostly is, a test costs about half of a try_wait)
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        if (ok && !mbar_test_wait(bar, parity) && !mbar_wait(bar, parity)) ok = false;
        return ok;
    };

    if (warp < kMmaWarp) {
        // ================================================================ softmax: warp = head, lane = token
        const int t = warp >> 2, h = warp & 3;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(h * 32) << 16) + t * 256;
        const float sl2 = s.scale * kLog2e;
        uint32_t n_s = 0, n_u = 0;               // items of this tile / units so far
        for (int idx = blockIdx.x; idx < n_units && ok; idx += gridDim.x, ++n_u) {
            const int ln = n_u & 1;
            if (!wait(&sm.list_full[ln], (n_u >> 1) & 1)) break;
            const int n = sm.n_tile[ln][t];
            const int blk = sm.blk[ln], pair = sm.pair[ln], b = sm.seq[ln], gk = pair - b * s.Hkv;
            const int tok = blk * kUnitTok + t * kTok + lane;
            const bool live = tok < a.n_tok;
            const int pos = lane_position(s, tok, a.n_tok), lc = local_lo(pos, s.W, kS) / kS;
            const float* bias = a.bias ? a.bias + (static_cast<long long>(b) * s.Hl + gk) * s.C : nullptr;
            float ref = kLowestLogit, den = 0.f;
            bool s_ready = false;
            int2 next = n > 0 ? sm.titem[ln][t][0] : make_int2(0, 0);
            for (int i = 0; i < n; ++i) {
                const int c = next.x;
                const uint32_t who = static_cast<uint32_t>(next.y);
                if (i + 1 < n) next = sm.titem[ln][t][i + 1];
                const float bb = (bias && c < lc) ? bias[c] : 0.f;
                const bool local = c >= lc;
                const bool act = ((who >> lane) & 1u) != 0u;
                if (!s_ready && !wait(&sm.s_full[t], n_s & 1)) break;
                __syncwarp();                        // (s_ready is a lane's own answer, and the loads take the whole warp)
                tc_fence_after_sync();
                float v[64], lm4[4];
                tmem_ld64_4(t_lane, t_lane + 64, v, lm4);
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.s_empty[t]);
                const int lim = local ? pos - c * kS : kS - 1;           // last visible key
                if (__any_sync(kFullMask, lim < kS - 1)) {
#pragma unroll
                    for (int j = 0; j < 64; ++j)
                        if (j > lim) v[j] = -INFINITY;
                }
                float mx[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                for (int j = 4; j < 60; j += 8) {
                    mx[0] = fmax3(mx[0], v[j], v[j + 1]);
                    mx[1] = fmax3(mx[1], v[j + 2], v[j + 3]);
                    mx[2] = fmax3(mx[2], v[j + 4], v[j + 5]);
                    mx[3] = fmax3(mx[3], v[j + 6], v[j + 7]);
                }
                mx[0] = fmax3(mx[0], v[60], v[61]);
                mx[1] = fmax3(mx[1], v[62], v[63]);
                float m = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                if (m == -INFINITY) m = 0.f;                             // no visible key (the row gets weight zero)
                const float2 sl22 = make_float2(sl2, sl2), nms2 = make_float2(-m * sl2, -m * sl2);
                float2 zp[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float2 x = __ffma2_rn(make_float2(v[2 * j], v[2 * j + 1]), sl22, nms2);
                    if ((j & 3) == 3) {
                        const float2 y = ex2_fma(x);
                        v[2 * j] = y.x;
                        v[2 * j + 1] = y.y;
                    } else {
                        v[2 * j] = ex2_approx(x.x);
                        v[2 * j + 1] = ex2_approx(x.y);
                    }
                    zp[j & 3] = __fadd2_rn(zp[j & 3], make_float2(v[2 * j], v[2 * j + 1]));
                }
                // (asked here, needed below: the answer arrives under the arithmetic)
                const bool o_ready = i == 0 || mbar_test_wait(&sm.o_done[t], (n_s - 1) & 1);
                const float2 z2 = __fadd2_rn(__fadd2_rn(zp[0], zp[1]), __fadd2_rn(zp[2], zp[3]));
                const float z = z2.x + z2.y;
                const float lam = local ? m * s.scale + __logf(z) : lm4[0] * s.scale + bb;
                // mixing weight relative to the row's reference
                float grow = 1.f;
                if (act && lam > ref + kRaise) {
                    grow = __expf(ref - lam);                            // (0 for the row's first chunk)
                    den *= grow;
                    ref = lam;
                }
                const float w = act ? __expf(lam - ref) : 0.f;
                den += w;
                const float qz = quotient(w, z), pw = act ? qz : 0.f;
                const float2 pw2 = make_float2(pw, pw);
                // the previous chunk's value product has read its probabilities and left the accumulator
                if (i > 0) {
                    if (!o_ready && !wait(&sm.o_done[t], (n_s - 1) & 1)) break;
                    __syncwarp();
                    if (__any_sync(kFullMask, grow != 1.f)) {
                        tc_fence_after_sync();
#pragma unroll 1
                        for (int cc = 0; cc < kD; cc += 16) {
                            float o[16];
                            tmem_ld16(t_lane + kOCol + cc, o);
                            uint32_t r0[8], r1[8];
#pragma unroll
                            for (int x = 0; x < 8; ++x) { r0[x] = __float_as_uint(o[x] * grow); r1[x] = __float_as_uint(o[8 + x] * grow); }
                            tmem_st8(t_lane + kOCol + cc, r0);
                            tmem_st8(t_lane + kOCol + cc + 8, r1);
                        }
                    }
                }
#pragma unroll
                for (int pc = 0; pc < 4; ++pc) {
                    uint32_t pk[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float2 p = __fmul2_rn(make_float2(v[pc * 16 + 2 * j], v[pc * 16 + 2 * j + 1]), pw2);
                        pk[j] = pack_bf16(p.x, p.y);
                    }
                    tmem_st8(t_lane + kPCol + pc * 8, pk);
                }
                s_ready = i + 1 < n && mbar_test_wait(&sm.s_full[t], (n_s + 1) & 1);
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.p_full[t]);
                ++n_s;
            }
            if (!ok) break;
            if (n > 0) {
                // ---- the tile's output rows
                if (!wait(&sm.o_done[t], (n_s - 1) & 1)) break;
                __syncwarp();
                tc_fence_after_sync();
                const float inv = live ? 1.f / den : 0.f;
                const long long orow = (static_cast<long long>(b) * s.Hq + gk * kG + h) * s.R + tok;
                const bool whole = blk * kUnitTok + t * kTok + kTok <= a.n_tok;
                // 64 dimensions at a time through the warp's own staging rows (not through the query tile: the next unit's queries
                // are on their way into it)
                uint8_t* stg = stage + warp * kStgBytes;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint4 w[8];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint32_t v[32];
                        tmem_ld32_issue(t_lane + kOCol + half * 64 + q * 32, v);
                        tmem_ld_wait32(v);
#pragma unroll
                        for (int pc = 0; pc < 4; ++pc) {
                            w[4 * q + pc].x = pack_bf16(__uint_as_float(v[8 * pc]) * inv, __uint_as_float(v[8 * pc + 1]) * inv);
                            w[4 * q + pc].y = pack_bf16(__uint_as_float(v[8 * pc + 2]) * inv, __uint_as_float(v[8 * pc + 3]) * inv);
                            w[4 * q + pc].z = pack_bf16(__uint_as_float(v[8 * pc + 4]) * inv, __uint_as_float(v[8 * pc + 5]) * inv);
                            w[4 * q + pc].w = pack_bf16(__uint_as_float(v[8 * pc + 6]) * inv, __uint_as_float(v[8 * pc + 7]) * inv);
                        }
                    }
                    if (whole) {
                        if (lane == 0) bulk_wait_read<0>();              // (the store before)
                        __syncwarp();
#pragma unroll
                        for (int pc = 0; pc < 8; ++pc) *reinterpret_cast<uint4*>(stg + swz128(lane, pc)) = w[pc];
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(&map_out, stg, half * 64, static_cast<int>(orow), l2_policy_evict_first());
                            bulk_commit();
                        }
                    } else if (live) {
#pragma unroll
                        for (int pc = 0; pc < 8; ++pc) *reinterpret_cast<uint4*>(a.out + orow * kD + half * 64 + pc * 8) = w[pc];
                    }
                    __syncwarp();                    // (the next half's loads take the whole warp)
                }
                tc_fence_before_sync();
                if (live) a.lse[orow] = ref + __logf(den);
            }
            if (a.write_sel && h == 0 && live) {
                int32_t* sel = a.sel + (static_cast<long long>(pair) * s.R + tok) * s.K;
                for (int x = 0; x < s.K; ++x) sel[x] = x < lc ? x : -1;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.list_empty[ln]);
        }
        if (lane == 0) bulk_wait_read<0>();
    } else if (warp < kLoadWarp) {
        // ================================================================ MMA issuer of tile t
        {
            const int t = warp - kMmaWarp;
            // (one answer per warp: elections follow)
            auto wait = [&](uint64_t* bar, uint32_t parity) {
                if (ok && !__all_sync(kFullMask, mbar_test_wait(bar, parity)) && !__all_sync(kFullMask, mbar_wait(bar, parity))) ok = false;
                return ok;
            };
            constexpr uint32_t idesc_s = umma_idesc_bf16(kRows, kNS);
            constexpr uint32_t idesc_o = umma_idesc_bf16(kRows, kD) | kUmmaBMnMajor;
            const uint32_t qa = smem_u32(qbuf + t * kQBytes), s_tm = tmem_base + t * 256;
            uint32_t g0 = 0, n_s = 0, n_p = 0, n_q = 0, n_u = 0;         // first item of the unit; scores, products, query tiles so far
            for (int idx = blockIdx.x; idx < n_units && ok; idx += gridDim.x, ++n_u) {
                const int ln = n_u & 1;
                if (!wait(&sm.list_full[ln], (n_u >> 1) & 1)) break;
                const int n = sm.n_items[ln];
                int left = sm.n_tile[ln][t];                             // scores of this tile still to be issued
                bool have_q = false, first = true;
                int issued = -1;                                         // last item whose scores were issued
                auto issue_s = [&](int i) {
                    const uint32_t st = (g0 + i) % kStages;
                    if (!have_q) { wait(&sm.q_full[t], n_q & 1); ++n_q; have_q = true; }
                    wait(&sm.kv_full[st], ((g0 + i) / kStages) & 1);
                    if (n_s > 0) wait(&sm.s_empty[t], (n_s - 1) & 1);
                    if (!ok) return;
                    tc_fence_after_sync();
                    const uint32_t ka = smem_u32(kbuf + st * kKBytes);
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            umma_bf16(s_tm, umma_desc_k128(qa + (ks >> 2) * 16384 + (ks & 3) * 32),
                                      umma_desc_k128(ka + (ks >> 2) * (kNS * 128) + (ks & 3) * 32), idesc_s, ks > 0 ? 1u : 0u);
                        umma_commit(&sm.s_full[t]);
                        if (left == 1) umma_commit(&sm.q_empty[t]);      // the next unit's queries may come
                    }
                    __syncwarp();
                    --left;
                    ++n_s;
                    issued = i;
                };
                for (int i = 0; i < n && ok; ++i) {
                    const uint32_t st = (g0 + i) % kStages;
                    if (!((sm.list[ln][i] >> (16 + t)) & 1)) {
                        // not this tile's: hand the buffers back (once they are there: the barrier's phase is theirs then)
                        if (wait(&sm.kv_full[st], ((g0 + i) / kStages) & 1) && lane == 0) mbar_arrive(&sm.kv_empty[st]);
                        continue;
                    }
                    if (issued < i) issue_s(i);
                    if (ok && i + 1 < n && ((sm.list[ln][i + 1] >> (16 + t)) & 1)) issue_s(i + 1);
                    if (!ok || !wait(&sm.p_full[t], n_p & 1)) break;
                    tc_fence_after_sync();
                    const uint32_t va = smem_u32(vbuf + st * kVBytes);
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            umma_bf16_ts(s_tm + kOCol, s_tm + kPCol + ks * 8, umma_desc_mn128(va + ks * 2048, 8192u, 1024u), idesc_o,
                                         (ks > 0 || !first) ? 1u : 0u);
                        umma_commit(&sm.kv_empty[st]);
                        umma_commit(&sm.o_done[t]);
                    }
                    __syncwarp();
                    first = false;
                    ++n_p;
                }
                g0 += static_cast<uint32_t>(n);
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.list_empty[ln]);
            }
        }
    } else if (warp == kLoadWarp) {
        // ================================================================ loader (one thread)
        if (lane == 0) {
            uint32_t g = 0, n_u = 0, n_q[2] = {0, 0};
            for (int idx = blockIdx.x; idx < n_units && ok; idx += gridDim.x, ++n_u) {
                const int ln = n_u & 1;
                int blk, pair;
                unit_of(idx, blk, pair);
                const int b = pair / s.Hkv, gk = pair - b * s.Hkv;
                auto load_q = [&] {
                    for (int t = 0; t < 2 && ok; ++t) {
                        if (blk * kUnitTok + t * kTok >= a.n_tok) continue;       // (a token attends its own chunk at least)
                        if (n_q[t] > 0 && !wait(&sm.q_empty[t], (n_q[t] - 1) & 1)) break;
                        mbar_expect_tx(&sm.q_full[t], kQBytes);
                        for (int h = 0; h < kG; ++h) {
                            const int row = (b * s.Hq + gk * kG + h) * s.R + blk * kUnitTok + t * kTok;
                            tma_load_2d(qbuf + t * kQBytes + h * 4096, &map_q, &sm.q_full[t], 0, row);
                            tma_load_2d(qbuf + t * kQBytes + 16384 + h * 4096, &map_q, &sm.q_full[t], 64, row);
                        }
                        ++n_q[t];
                    }
                };
                if (n_u == 0) load_q();                                  // (under the making of the first list)
                if (!ok || !wait(&sm.list_full[ln], (n_u >> 1) & 1)) break;
                const int n = sm.n_items[ln], base = sm.base[ln];
                auto load_item = [&](int i) {
                    const uint32_t st = g % kStages;
                    const int c = base + (sm.list[ln][i] & 0xffff);
                    if (g >= kStages && !wait(&sm.kv_empty[st], ((g / kStages) - 1) & 1)) return;
                    const int row = c * kS;
                    // chunks left of every token's window have a landmark row (the others' score column is not used)
                    const bool lm = c < s.C;
                    uint8_t* kd = kbuf + st * kKBytes;
                    mbar_expect_tx(&sm.kv_full[st], 16384 + kVBytes + (lm ? 256 : 0));
                    tma_load_3d(kd, &map_k, &sm.kv_full[st], 0, row, pair);
                    tma_load_3d(kd + kNS * 128, &map_k, &sm.kv_full[st], 64, row, pair);
                    if (lm) {
                        // row 64: its 16-byte pieces stay in place under the swizzle (64 mod 8 = 0)
                        const __nv_bfloat16* src = a.lm + ((static_cast<long long>(b) * s.Hl + gk) * s.C + c) * kD;
                        bulk_load(kd + 64 * 128, src, 128, &sm.kv_full[st]);
                        bulk_load(kd + kNS * 128 + 64 * 128, src + 64, 128, &sm.kv_full[st]);
                    }
                    tma_load_3d(vbuf + st * kVBytes, &map_v, &sm.kv_full[st], 0, row, pair);
                    tma_load_3d(vbuf + st * kVBytes + 8192, &map_v, &sm.kv_full[st], 64, row, pair);
                    ++g;
                };
                // in the order in which the buffers become free: the first chunk's, the queries' with the last unit's last scores
                int i = 0;
                if (n > 0) load_item(i++);
                if (n_u > 0) load_q();
                for (; i < n && ok; ++i) load_item(i);
                mbar_arrive(&sm.list_empty[ln]);
            }
            // own copies in flight must have landed before the CTA leaves
            for (uint32_t k = g > kStages ? g - kStages : 0; k < g; ++k) mbar_wait(&sm.kv_full[k % kStages], (k / kStages) & 1);
        }
    } else {
        // ================================================================ the unit's chunk list, one unit ahead
        uint32_t n_u = 0, n_ids = 0;
        for (int idx = blockIdx.x; idx < n_units && ok; idx += gridDim.x, ++n_u) {
            int blk, pair;
            unit_of(idx, blk, pair);
            const int ln = n_u & 1;
            if (n_u >= 2 && !wait(&sm.list_empty[ln], ((n_u >> 1) - 1) & 1)) break;
            const int tok0 = blk * kUnitTok;
            const int last = s.pos0 + min(a.n_tok, tok0 + kUnitTok) - 1;
            const int base = a.local ? local_lo(s.pos0 + tok0, s.W, kS) / kS : 0, n_vis = last / kS + 1 - base;
            // The first list of a CTA is waited for, and its instructions come from memory: short loops.  (2 x 6000 tokens, K = 32, cycles:
            // an atomic in shared memory per selected chunk 13000 - 26000, bits per token turned by votes, unrolled, 28000.)
            const bool picks = !a.local && local_lo(last, s.W, kS) / kS > s.K;       // some token has more candidates than places
            if (picks) {
                for (int c = lane; c < n_vis; c += 32) { sm.mask[0][c] = 0u; sm.mask[1][c] = 0u; }
                __syncwarp();
                // the selections of 64 (32 where they are long) tokens at a time
                const int step = s.K <= 32 ? kUnitTok : kTok;
#pragma unroll 1
                for (int x0 = 0; x0 < kUnitTok; x0 += step) {
                    const int nx = min(step, a.n_tok - tok0 - x0), words = nx * s.K;
                    if (nx <= 0) break;
                    const int32_t* sel = a.sel + (static_cast<long long>(pair) * s.R + tok0 + x0) * s.K;
                    if (((reinterpret_cast<uintptr_t>(sel) | static_cast<uintptr_t>(4 * words)) & 15) == 0) {
                        if (lane == 0) {
                            mbar_expect_tx(&sm.ids_full, 4 * words);
                            bulk_load(sm.ids, sel, 4 * words, &sm.ids_full);
                        }
                        __syncwarp();
                        if (!wait(&sm.ids_full, n_ids++ & 1)) break;
                    } else {
#pragma unroll 8
                        for (int y = lane; y < words; y += 32) sm.ids[y] = sel[y];
                    }
                    __syncwarp();
                    // lane = token, which starts at its own slot: neighbours' slots lie K words apart
#pragma unroll 1
                    for (int y0 = 0; y0 < nx; y0 += kTok) {
                        const int32_t* id = sm.ids + (y0 + lane) * s.K;
                        uint32_t* mask = sm.mask[(x0 + y0) / kTok];
                        if (y0 + lane < nx) {
                            int e = lane % s.K;
#pragma unroll 4
                            for (int i = 0; i < s.K; ++i) {
                                const int c = id[e];
                                if (c >= 0 && c < n_vis) atomicOr(mask + c, 1u << lane);
                                e = e + 1 < s.K ? e + 1 : 0;
                            }
                        }
                        __syncwarp();
                    }
                    // The next rows may come the other way: ordinary accesses to sm.ids are ordered before a bulk copy into it by a proxy
                    // fence of the lane that made them alone.  (One CTA meets both ways where top_k is no multiple of 4.)
                    fence_proxy_async_smem();
                    __syncwarp();
                }
                if (!ok) break;
            }
            int n = 0, nt[2] = {0, 0};
#pragma unroll 1
            for (int c0 = 0; c0 < n_vis; c0 += 32) {
                const int c = c0 + lane;
                const uint32_t below = (1u << lane) - 1u;
                uint32_t m[2];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    // token x of the tile sees chunk c from x = own on, and as a candidate (left of its window) from x = left on
                    const int first = s.pos0 + tok0 + t * kTok, own = (base + c) * kS - first, left = (base + c + 1) * kS + s.W - 1 - first;
                    const uint32_t live = bits_below(a.n_tok - tok0 - t * kTok), seen = ~bits_below(own), cand = ~bits_below(left);
                    m[t] = c < n_vis ? live & ((seen & ~cand) | (a.local ? 0u : picks ? sm.mask[t][c] : cand)) : 0u;
                    const unsigned v = __ballot_sync(kFullMask, m[t] != 0u);
                    if (m[t]) sm.titem[ln][t][nt[t] + __popc(v & below)] = make_int2(base + c, static_cast<int>(m[t]));
                    nt[t] += __popc(v);
                }
                const unsigned v = __ballot_sync(kFullMask, (m[0] | m[1]) != 0u);
                if (m[0] | m[1]) sm.list[ln][n + __popc(v & below)] = c | (m[0] ? 1 << 16 : 0) | (m[1] ? 1 << 17 : 0);
                n += __popc(v);
            }
            if (lane == 0) {
                sm.blk[ln] = blk;
                sm.pair[ln] = pair;
                sm.seq[ln] = pair / s.Hkv;
                sm.n_items[ln] = n;
                sm.base[ln] = base;
                sm.n_tile[ln][0] = nt[0];
                sm.n_tile[ln][1] = nt[1];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.list_full[ln]);
        }
    }
    if (!ok && lane == 0) set_status(a.status, kDevTimeout);
    __syncwarp();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == kMmaWarp) tmem_dealloc(tmem_base, 512);
}

}  // namespace

// Tokens of a call (from its first on) that go this way: a multiple of 128 below the call's length, or all of them.  The
// split with the largest gain by these costs (SM cycles; fitted to 16K, 2 x 6000 and 3 x 1000 tokens):
//   here, a unit of 64 tokens: 2200 per chunk it visits (at most every visible one) + 12000, the last unit at least in full;
//   chunk-major (index, attend and fuse kernels): 3830 per 32 tokens and chunk they attend, and 50000 for the launches (which rest on one
//   pair: 2 KV heads, K = 16, us all here / all chunk-major 3000 tokens 70 / 72, 4000 tokens 88 / 84).
// With units for every SM the line lies near visible : attended = 5 : 2.  With few (sequence, KV head) pairs the units are a
// serial chain on some of the SMs, and everything goes chunk-major unless that saves its launches (2 KV heads, a slice of
// 2190 tokens at 4395, K = 32: 107 us chunk-major, 193 with the first 768 tokens here).  The parts of a call that the library
// itself cuts into slices keep the whole call's split (Shape::qsplit): the same bits either way.
int prefill_query_tokens(const Shape& s) {
    if (s.Hl != s.Hkv || s.K > kMaxK) return 0;
    if (s.qsplit >= 0) {
        const int n = s.qsplit - s.pos0;
        return n <= 0 ? 0 : n >= s.R ? s.R : n / 128 * 128;
    }
    const int nl = (s.W - 1 + kS - 1) / kS + 1;                          // chunks of a local window
    const long long pairs = static_cast<long long>(s.B) * s.Hkv, sms = sm_count();
    long long here = 0, there = 0, most = 0;
    int best = 0;
    for (int n = 0; n < s.R;) {
        const int end = n + kUnitTok < s.R ? n + kUnitTok : s.R;
        const long long vis = (s.pos0 + end - 1) / kS + 1, att = vis < s.K + nl ? vis : s.K + nl, unit = 2200 * vis + 12000;
        if (vis > kMaxC) break;
        here += pairs * unit;
        there += pairs * (end - n) * att * 3830 / 32;
        n = end;
        const long long t = here / sms > unit ? here / sms : unit, gain = there / sms + (n == s.R ? 50000 : 0) - t;
        if (gain > most && (n == s.R || n % 128 == 0)) {
            most = gain;
            best = n;
        }
    }
    return best;
}

// Whether the local windows of the chunk-major tokens (from `first` on) go this way too, as one partial output row per token
// and head (in out and lse, for the fuse kernel) instead of one per window chunk.  SM cycles: a unit visits the nl chunks of a window
// and one more, 2200 each + 6000, in rounds of a unit per SM, and the launch takes 15000; chunk-major 3400 per 32 tokens and window chunk
// (their lists are long).  Measured, us chunk-major / here: 16K tokens, K = 16, W = 64 934 / 941, 128 978 / 955, 256 1047 / 978; K = 32,
// W = 512 1567 / 1403; a slice of 2048 tokens at 48K, K = 32, W = 128 331 / 332, 256 329 / 327, 512 356 / 332; of 300 tokens 71 / 75.
bool prefill_local_query(const Shape& s, int first) {
    if (s.Hl != s.Hkv) return false;
    if (s.lsplit >= 0) return s.lsplit != 0;
    const int nl = (s.W - 1 + kS - 1) / kS + 1;
    const long long pairs = static_cast<long long>(s.B) * s.Hkv, sms = sm_count(), toks = s.R - first;
    const long long rounds = (pairs * ((toks + kUnitTok - 1) / kUnitTok) + sms - 1) / sms;
    return rounds * (2200 * (nl + 1) + 6000) + 15000 < pairs * toks * nl * 3400 / 32 / sms;
}

int launch_prefill_query_tc(const Shape& s, const Tensors& t, int first, int n_tok, int local, int write_sel, cudaStream_t stream) {
    const uint64_t pairs = static_cast<uint64_t>(s.B) * s.Hkv, q_rows = static_cast<uint64_t>(s.B) * s.Hq * s.R;
    CUtensorMap map_q, map_k, map_v, map_out;
    if (!make_bf16_2d_map(&map_q, t.q, q_rows, kD, 64, kTok) || !make_kv_map(&map_k, t.k, pairs, s.T, s.pos0 + s.R, kD, 64, kS) ||
        !make_kv_map(&map_v, t.v, pairs, s.T, s.pos0 + s.R, kD, 64, kS) || !make_bf16_2d_map(&map_out, t.out, q_rows, kD, 64, kTok))
        return HILS_ERR_CUDA;
    const size_t smem = kStages * (kKBytes + kVBytes) + 2 * kQBytes + kMmaWarp * kStgBytes + sizeof(QmSmem) + 1024;
    static PerDeviceOnce once;
    if (once.pending()) {
        if (cudaFuncSetAttribute(prefill_query_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
            return HILS_ERR_CUDA;
        once.done();
    }
    QmArgs a{s, static_cast<const __nv_bfloat16*>(t.landmarks), t.bias, t.sel_idx, static_cast<__nv_bfloat16*>(t.out), t.lse, t.status,
             first, n_tok, local, write_sel};
    const long long units = static_cast<long long>(s.B) * s.Hkv * ((n_tok - first + kUnitTok - 1) / kUnitTok);
    const unsigned grid = static_cast<unsigned>(units < sm_count() ? units : sm_count());
    if (launch_pdl(prefill_query_tc_kernel, dim3(grid), dim3(kThreads), smem, stream, map_q, map_k, map_v, map_out, a) != cudaSuccess)
        return HILS_ERR_CUDA;
    return 1;
}

}  // namespace hils
