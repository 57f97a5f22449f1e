// Landmark scoring + exact top-K for prefill on the 5th-generation tensor cores (tcgen05 + TMEM).
//
// One persistent CTA per SM walks (sequence, KV head, 128-token tile) triples, heavy tiles first.  The tile's queries
// (4 heads x 128 tokens x 128 d) stay in shared memory; landmark tiles of 64 chunks stream through a TMA ring.  One warp
// issues tcgen05.mma (M = 128 tokens, N = 64 chunks, K = 128) once per head into tensor memory, double buffered.
// Scan warps own one token per thread (token = TMEM lane): they read the four heads' scores, take the group max (App. C)
// and append the candidates that beat the token's K-th best score known so far to a buffer in shared memory, in arrival
// order = ascending chunk id.  When a buffer of the warp may fill up it goes to the warp's partner among the sort warps,
// and the scan goes on with the other buffer.  The sort warp keeps the token's exact running top-K (Eq. surrogate top-k;
// equal scores go to the lower chunk id): the N best SCORES so far stay sorted in registers; it sorts the new ones
// (register network on 32-bit values: one max and one min per compare-exchange), merges them in, reads the new K-th best
// score off the list, and filters the kept entries in place: everything above that score and the earliest of those equal
// to it, exactly K, still in ascending chunk order -- the order in which it writes the selection at the end of the tile,
// while the scan works on the next one.  The number of buffers grows with log(candidates / K), not with the candidates.
// Bound: the latencies of the sort warps' code (one per scheduler; with scan and sort in one warp 16K tokens, K = 16 took
// 101.5 us instead of 95, a 2048-token slice at 48K, K = 32, 74 instead of 68).
#include "internal.h"
#include "tma.cuh"

namespace hils {
namespace {

constexpr int kD = 128;
constexpr int kS = 64;
constexpr int kG = 4;
constexpr int kTileTok = 128;
constexpr int kLmStages = 2;
constexpr int kLmStageBytes = kS * kD * 2;          // 64 landmark rows = two 8 KB K-blocks
constexpr int kQBytes = kG * kTileTok * kD * 2;     // 128 KB
constexpr int kMaxK = 32;
constexpr int kRoom = 16;                           // candidates that a thread hands over at a time
constexpr int kTmaWarp = 4, kMmaWarp = 5, kSortWarp = 6;
constexpr int kThreads = 320;                       // 4 scan warps, 1 TMA warp, 1 MMA warp, 4 sort warps
constexpr uint32_t kTmemCols = 512;                 // 2 buffers x 4 heads x 64 columns

struct TcArgs {
    Shape s;
    const float* bias;
    int32_t* sel;
    int* status;
    // optional: per-(query block, pair, chunk) counts of the (token, slot) entries that attend each chunk -- the
    // first step of the inverse index, taken here because the selections are at hand (NULL: not wanted)
    int* cnt;
    int qb, nc, t0;    // tokens per query block (a multiple of the 128-token tile), chunk slots per pair in cnt, first token counted
    int local;         // 1: the chunks of the local windows are counted too
};

struct TcSmem {
    uint64_t q_empty;          // every MMA of the tile has completed: its query tile may be overwritten
    uint64_t q_full;
    uint64_t full[kLmStages];
    uint64_t empty[kLmStages];
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint32_t tmem_base;
    int abort;                 // a bounded wait of a sort warp ran out: every sort warp leaves after the tile
    uint64_t new_full[4][2], new_empty[4][2];   // [scan warp][buffer] candidates handed over / read
    int last[2][4];                             // the buffer is its tile's last
    uint8_t n_new[2][kTileTok];                 // candidates of each thread
    float tau[2][kTileTok];                     // [tile parity] each token's K-th best score so far
};

// Sorts N scores in registers, largest first (Batcher's odd-even merge sort, fully unrolled: static register
// indices; a compare-exchange is one max and one min; 191 of them for 32 scores, a bitonic network takes 240).
template <int N>
__device__ __forceinline__ void oddeven_sort_desc(float (&a)[N]) {
    constexpr int kLog = N == 32 ? 5 : 4;
#pragma unroll
    for (int ps = 0; ps < kLog; ++ps) {
#pragma unroll
        for (int ks = kLog - 1; ks >= 0; --ks) {
            if (ks > ps) continue;
            const int p = 1 << ps, k = 1 << ks;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                // pairs (i, i + k) with i - k % p in the lower half of a block of 2 k, both in one block of 2 p
                const int r = i - k % p;
                if (r >= 0 && (r & k) == 0 && i + k < N && i / (2 * p) == (i + k) / (2 * p)) {
                    const float hi = fmaxf(a[i], a[i + k]), lo = fminf(a[i], a[i + k]);
                    a[i] = hi;
                    a[i + k] = lo;
                }
            }
        }
    }
}
// Sorts a bitonic sequence of N scores, largest first.
template <int N>
__device__ __forceinline__ void bitonic_merge_desc(float (&a)[N]) {
    constexpr int kLog = N == 32 ? 5 : 4;
#pragma unroll
    for (int js = kLog - 1; js >= 0; --js) {
        const int j = 1 << js;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int l = i ^ j;
            if (l > i) {
                const float hi = fmaxf(a[i], a[l]), lo = fminf(a[i], a[l]);
                a[i] = hi;
                a[l] = lo;
            }
        }
    }
}

// Entries are compacted by storing each where the kept ones end so far and moving the end only if it is kept.  The addresses are
// worked out before the stores, each in a register of its own: an address that is advanced behind its store waits until the store
// has read it (34 cycles per candidate, 2170 of a step's 6230; the stores' predicates and the kept entries' filter the same).
__device__ __forceinline__ void st_entry(uint32_t at, uint32_t chunk, float score) {
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(chunk), "r"(__float_as_uint(score)) : "memory");
}
__device__ __forceinline__ void st_entry(uint32_t at, unsigned long long raw) { asm volatile("st.shared.b64 [%0], %1;" ::"r"(at), "l"(raw) : "memory"); }

// N = length of the per-token sorted score list: 16 for K <= 16, else 32.
// PERHEAD: one landmark row (and bias) per query head (App. C) instead of one per KV head.  A template parameter, not
// a run-time branch: the scan loop's code has to stay small (the kernel is sensitive to instruction fetch).
template <int N, bool PERHEAD>
__global__ void __launch_bounds__(kThreads, 1)
prefill_select_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_lm,
                         const TcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* qs = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* lms = qs + kQBytes;
    unsigned long long* lists = reinterpret_cast<unsigned long long*>(lms + kLmStages * kLmStageBytes);   // [2 kMaxK][128]
    TcSmem& sm = *reinterpret_cast<TcSmem*>(lists + 2 * kMaxK * kTileTok);

    const Shape& s = a.s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pairs = s.B * s.Hkv;
    const int tiles_per_seq = (s.R + kTileTok - 1) / kTileTok;
    const int n_tiles = pairs * tiles_per_seq;
    const int K = s.K;
    constexpr int per = PERHEAD ? kG : 1;     // landmark rows per chunk
    // A CTA walks the tiles blockIdx.x, blockIdx.x + gridDim.x, ... (heavy tiles first): the query tile and the first
    // scores of the next tile are fetched and computed while the sort warps still finish the previous one.  Every
    // role derives the same tile sequence; tiles without candidates touch no barrier.
    // (Every other round of the walk runs backwards, so that a CTA early in one round, with heavy tiles, is late in the next.)
    auto tile_of = [&](int idx, int& ti, int& pair, int& nsteps) {
        const int rnd = idx / static_cast<int>(gridDim.x);
        if (rnd & 1) idx = min(n_tiles, (rnd + 1) * static_cast<int>(gridDim.x)) - 1 - (idx - rnd * static_cast<int>(gridDim.x));
        ti = tiles_per_seq - 1 - idx / pairs;
        pair = idx % pairs;
        // candidates of a token = the chunks left of its local window (Sec. 2.1); the tile's last token has the most
        const int last_tok = min(s.R, (ti + 1) * kTileTok) - 1;
        const int ncand_max = local_lo(s.pos0 + last_tok, s.W, kS) / kS;
        nsteps = ncand_max <= K ? 0 : (ncand_max + kS - 1) / kS;        // (up to K candidates: all of them, no scores needed)
    };

    if (tid == 0) {
        mbar_init(&sm.q_full, 1);
        mbar_init(&sm.q_empty, 1);
        sm.abort = 0;
        for (int i = 0; i < kLmStages; ++i) { mbar_init(&sm.full[i], 1); mbar_init(&sm.empty[i], 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.tmem_full[i], 1);
            mbar_init(&sm.tmem_empty[i], 4);
            for (int w = 0; w < 4; ++w) { mbar_init(&sm.new_full[w][i], 1); mbar_init(&sm.new_empty[w][i], 1); }
        }
        mbar_fence_init();
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_lm);
    }
    if (warp == kMmaWarp) tmem_alloc(&sm.tmem_base, kTmemCols);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = sm.tmem_base;
    pdl_wait();

    if (warp == kTmaWarp) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t n_lm = 0;            // landmark tiles requested so far, over all tiles of this CTA
            int tn = 0;                   // tiles with candidates so far
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_tiles && ok; idx += gridDim.x) {
                int ti, pair, nsteps;
                tile_of(idx, ti, pair, nsteps);
                if (nsteps == 0) continue;
                const int b = pair / s.Hkv, gk = pair % s.Hkv;
                if (tn > 0) ok = mbar_wait(&sm.q_empty, (tn - 1) & 1);
                if (!ok) break;
                mbar_expect_tx(&sm.q_full, kQBytes);
                for (int h = 0; h < kG; ++h) {
                    const int row = (b * s.Hq + gk * kG + h) * s.R + ti * kTileTok;
                    tma_load_2d(qs + h * 32768, &map_q, &sm.q_full, 0, row);
                    tma_load_2d(qs + h * 32768 + 16384, &map_q, &sm.q_full, 64, row);
                }
                // landmark tiles in ring order: step it, landmark head hh (per = 1: one tile per step for all heads;
                // per = G: one tile per query head, App. C)
                const int ntiles = nsteps * per;
                for (int n = 0; n < ntiles && ok; ++n, ++n_lm) {
                    const int st = n_lm % kLmStages, it = n / per, hh = n % per;
                    if (n_lm >= kLmStages) ok = mbar_wait(&sm.empty[st], ((n_lm / kLmStages) - 1) & 1);
                    if (!ok) break;
                    uint8_t* dst = lms + st * kLmStageBytes;
                    const int row = ((b * s.Hl + gk * per + hh)) * s.C + it * kS;
                    mbar_expect_tx(&sm.full[st], kLmStageBytes);
                    tma_load_2d(dst, &map_lm, &sm.full[st], 0, row);
                    tma_load_2d(dst + 8192, &map_lm, &sm.full[st], 64, row);
                }
                ++tn;
            }
            if (!ok) set_status(a.status, kDevTimeout);
            // own copies in flight: the last query tile and the last stages must have landed before exit
            if (tn > 0) mbar_wait(&sm.q_full, (tn - 1) & 1);
            for (uint32_t n = n_lm > kLmStages ? n_lm - kLmStages : 0; n < n_lm; ++n)
                mbar_wait(&sm.full[n % kLmStages], (n / kLmStages) & 1);
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------------ MMA issuer
        {
            // (one answer per warp: elections follow)
            auto wait = [](uint64_t* bar, uint32_t parity) { return __all_sync(kFullMask, mbar_wait(bar, parity)) != 0; };
            constexpr uint32_t idesc = umma_idesc_bf16(kTileTok, kS);
            // S_h = Q_h x landmark tile^T (M = 128 tokens, N = 64 chunks, K = 128) into head h's 64 columns
            auto issue_head = [&](uint32_t d_tmem, uint32_t q_addr, uint32_t lm_addr) {
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    const uint64_t da = umma_desc_k128(q_addr + (ks >> 2) * 16384 + (ks & 3) * 32);
                    const uint64_t db = umma_desc_k128(lm_addr + (ks >> 2) * 8192 + (ks & 3) * 32);
                    umma_bf16(d_tmem, da, db, idesc, ks > 0 ? 1u : 0u);
                }
            };
            const uint32_t q0 = smem_u32(qs);
            uint32_t n_lm = 0, n_step = 0;     // landmark tiles / steps so far, over all tiles of this CTA
            int tn = 0;
            bool ok = true;
            for (int idx = blockIdx.x; idx < n_tiles && ok; idx += gridDim.x) {
                int ti, pair, nsteps;
                tile_of(idx, ti, pair, nsteps);
                if (nsteps == 0) continue;
                ok = wait(&sm.q_full, tn & 1);
                for (int it = 0; it < nsteps && ok; ++it, ++n_step) {
                    const uint32_t buf = n_step & 1u;
                    if (n_step >= 2) ok = wait(&sm.tmem_empty[buf], ((n_step >> 1) - 1) & 1);
                    if (!ok) break;
                    if (per == 1) {
                        // one landmark tile for the four query heads
                        const uint32_t st = n_lm % kLmStages;
                        ok = wait(&sm.full[st], (n_lm / kLmStages) & 1);
                        if (!ok) break;
                        tc_fence_after_sync();
                        const uint32_t lm_addr = smem_u32(lms + st * kLmStageBytes);
                        if (elect_one()) {
#pragma unroll
                            for (int h = 0; h < kG; ++h) issue_head(tmem_base + buf * 256 + h * kS, q0 + h * 32768, lm_addr);
                            umma_commit(&sm.empty[st]);        // landmark stage reusable once these MMAs are done
                            umma_commit(&sm.tmem_full[buf]);   // scores of this step readable
                        }
                        __syncwarp();
                        ++n_lm;
                    } else {
                        // one landmark tile per query head (App. C), in ring order
#pragma unroll
                        for (int h = 0; h < kG; ++h) {
                            const uint32_t st = n_lm % kLmStages;
                            if (ok) ok = wait(&sm.full[st], (n_lm / kLmStages) & 1);
                            if (ok) {
                                tc_fence_after_sync();
                                if (elect_one()) {
                                    issue_head(tmem_base + buf * 256 + h * kS, q0 + h * 32768, smem_u32(lms + st * kLmStageBytes));
                                    umma_commit(&sm.empty[st]);
                                    if (h == kG - 1) umma_commit(&sm.tmem_full[buf]);
                                }
                                __syncwarp();
                                ++n_lm;
                            }
                        }
                        if (!ok) break;
                    }
                }
                if (ok && elect_one()) umma_commit(&sm.q_empty);          // the query tile may be replaced once all of these are done
                __syncwarp();
                ++tn;
            }
            if (!ok && lane == 0) set_status(a.status, kDevTimeout);
        }
    } else if (warp < kTmaWarp) {
        // ------------------------------------------------------------------ scan: one token per thread
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(warp * 32) << 16);
        const uint32_t room_at = smem_u32(lists) + tid * 8;      // [buffer][kRoom][128] entries
        uint32_t n_step = 0, n_buf = 0;                          // steps / buffers so far, over all tiles of this CTA
        int tn = 0;                                              // tiles with candidates so far
        bool ok = true;
        for (int idx = blockIdx.x; idx < n_tiles && ok; idx += gridDim.x) {
            int ti, pair, nsteps;
            tile_of(idx, ti, pair, nsteps);
            if (nsteps == 0) continue;
            const int b = pair / s.Hkv, gk = pair % s.Hkv;
            const int my_ncand = local_lo(s.pos0 + ti * kTileTok + tid, s.W, kS) / kS;
            // bias rows of this KV head's landmark heads (per = 1: one row, shared by the four query heads)
            const float* bias = a.bias ? a.bias + (static_cast<long long>(b) * s.Hl + gk * per) * s.C : nullptr;
            uint32_t at0 = 0, at = 0;
            auto acquire = [&]() {
                if (n_buf >= 2 && !__all_sync(kFullMask, mbar_wait(&sm.new_empty[warp][n_buf & 1], ((n_buf >> 1) - 1) & 1))) ok = false;
                at = at0 = room_at + (n_buf & 1) * (kRoom * 8 * kTileTok);
            };
            auto hand_over = [&](bool last) {
                sm.n_new[n_buf & 1][tid] = static_cast<uint8_t>((at - at0) / (8 * kTileTok));
                if (lane == 0) sm.last[n_buf & 1][warp] = last;
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.new_full[warp][n_buf & 1]);
                ++n_buf;
            };
            // (the sort warp has read the last buffer of the tile two before, so it writes this slot no more)
            acquire();
            volatile float* tau_sm = &sm.tau[tn & 1][tid];
            *tau_sm = -INFINITY;
            for (int it = 0; it < nsteps && ok; ++it, ++n_step) {
                const uint32_t buf = n_step & 1u;
                if (!__all_sync(kFullMask, mbar_wait(&sm.tmem_full[buf], (n_step >> 1) & 1))) { ok = false; break; }
                tc_fence_after_sync();
                const bool tail = (it + 1) * kS > my_ncand;     // only the last step holds chunks this token may not see
#pragma unroll 1
                for (int cb = 0; cb < 4; ++cb) {
                    float u16[16];
                    float r[4][16];
                    const uint32_t col = t_lane + buf * 256 + cb * 16;
                    tmem_ld16x4(col, col + kS, col + 2 * kS, col + 3 * kS, r);
                    const int cbase = it * kS + cb * 16;
                    if (PERHEAD && bias != nullptr) {
                        // every head adds its own bias before the maximum over the group (App. C)
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const int cc = min(cbase + j, s.C - 1);
                            u16[j] = fmaxf(fmaxf(fmaf(r[0][j], s.scale, bias[cc]), fmaf(r[1][j], s.scale, bias[s.C + cc])),
                                           fmaxf(fmaf(r[2][j], s.scale, bias[2 * s.C + cc]), fmaf(r[3][j], s.scale, bias[3 * s.C + cc]))) + 0.0f;
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) u16[j] = fmaf(fmaxf(fmax3(r[0][j], r[1][j], r[2][j]), r[3][j]), s.scale, 0.0f);   // (no -0)
                        if (bias) {
                            const float* bp = bias + cbase;
                            if (cbase + 16 <= s.C) {
#pragma unroll
                                for (int j = 0; j < 16; ++j) u16[j] += __ldg(bp + j);
                            } else {
#pragma unroll
                                for (int j = 0; j < 16; ++j) u16[j] += __ldg(bias + min(cbase + j, s.C - 1));
                            }
                        }
                    }
                    if (tail) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (cbase + j >= my_ncand) u16[j] = -INFINITY;
                    }
                    if (cb == 3) {
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sm.tmem_empty[buf]);
                    }
                    // Filter on the score: a candidate that only EQUALS the K-th best score so far loses to the K
                    // candidates at or above it, which all have lower chunk ids.  (The threshold may be some buffers old.)
                    const int c0 = it * kS + cb * 16;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (__any_sync(kFullMask, at - at0 > (kRoom - 8) * 8 * kTileTok)) {
                            hand_over(false);
                            acquire();
                        }
                        const float tau = *tau_sm;
                        uint32_t to[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {                    // (there is room for all eight)
                            to[j] = at;
                            at += u16[8 * h + j] > tau ? 8 * kTileTok : 0;
                        }
#pragma unroll
                        for (int j = 0; j < 8; ++j) st_entry(to[j], c0 + 8 * h + j, u16[8 * h + j]);
                    }
                }
            }
            if (ok) hand_over(true);
            ++tn;
        }
        if (!ok && lane == 0) set_status(a.status, kDevTimeout);
    } else {
        // ------------------------------------------------------------------ sort: one token per thread
        const int sw = warp - kSortWarp, row = sw * 32 + lane;
        unsigned long long* pool = lists + 2 * kRoom * kTileTok + row;       // the token's kept entries: entry e at pool[e * 128]
        const uint32_t pool_at = smem_u32(pool);
        uint32_t n_buf = 0;
        int tn = 0;
        bool ok = true;
        for (int idx = blockIdx.x; idx < n_tiles; idx += gridDim.x) {
        int ti, pair, nsteps;
        tile_of(idx, ti, pair, nsteps);
        const int tok = ti * kTileTok + row;
        const int my_ncand = local_lo(s.pos0 + tok, s.W, kS) / kS;
        float best[N];                     // the N best scores so far, largest first (-inf = none)
#pragma unroll
        for (int e = 0; e < N; ++e) best[e] = -INFINITY;
        int cnt = 0;
        for (bool last = nsteps == 0; !last && ok; ++n_buf) {
            const uint32_t bf = n_buf & 1u;
            if (!__all_sync(kFullMask, mbar_wait(&sm.new_full[sw][bf], (n_buf >> 1) & 1))) { ok = false; break; }
            const int n_new = sm.n_new[bf][row];
            last = sm.last[bf][sw] != 0;
            unsigned long long raw[kRoom];
            const unsigned long long* src = lists + bf * (kRoom * kTileTok) + row;
#pragma unroll
            for (int e = 0; e < kRoom; ++e) raw[e] = src[e * kTileTok];
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.new_empty[sw][bf]);
            // the N best scores of (best so far) + (new): sort the new ones, take the larger of the i-th best old and the
            // i-th worst new, sort that bitonic sequence
            float nw[kRoom];
            auto score = [&](int e) { return __uint_as_float(static_cast<uint32_t>(raw[e] >> 32)); };
#pragma unroll
            for (int e = 0; e < kRoom; ++e) nw[e] = e < n_new ? score(e) : -INFINITY;
            oddeven_sort_desc<kRoom>(nw);
#pragma unroll
            for (int e = 0; e < kRoom; ++e) best[N - 1 - e] = fmaxf(best[N - 1 - e], nw[e]);
            bitonic_merge_desc<N>(best);
            // the K-th best = the smallest of the first K (written so that the list stays in registers:
            // picking entry K - 1 would index it dynamically)
            float tau = INFINITY;
#pragma unroll
            for (int e = 0; e < N; ++e) tau = fminf(tau, e < K ? best[e] : INFINITY);
            if (!last) *const_cast<volatile float*>(&sm.tau[tn & 1][row]) = tau;
            // Exactly K survive: every score above tau, and the earliest of those equal to it.  All at or above it first;
            // that leaves more than K only where scores beyond the K-th equal it.
            // (eight entries per round: their loads go out together)
            uint32_t to = pool_at;
#pragma unroll 1
            for (int e0 = 0; e0 < cnt; e0 += 8) {
                unsigned long long old[8];
                uint32_t at[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) old[j] = pool[(e0 + j) * kTileTok];
#pragma unroll
                for (int j = 0; j < 8; ++j) {                           // (to <= the entry: in place, in order)
                    at[j] = to;
                    to += __uint_as_float(static_cast<uint32_t>(old[j] >> 32)) >= tau && e0 + j < cnt ? 8 * kTileTok : 0;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) st_entry(at[j], old[j]);
            }
            cnt = static_cast<int>(to - pool_at) / (8 * kTileTok);
            uint32_t live = 0;                                  // new entries that stay
#pragma unroll
            for (int e = 0; e < kRoom; ++e) live |= (e < n_new && score(e) >= tau) ? 1u << e : 0u;
            if (cnt + __popc(live) > K) {
                int above = 0;
#pragma unroll
                for (int e = 0; e < N; ++e) above += (e < K && best[e] > tau) ? 1 : 0;
                int ties = K - above, w = 0;
#pragma unroll 1
                for (int e = 0; e < cnt; ++e) {
                    const unsigned long long x = pool[e * kTileTok];
                    const bool tie = __uint_as_float(static_cast<uint32_t>(x >> 32)) == tau;
                    if (!tie || ties > 0) pool[w++ * kTileTok] = x;
                    ties -= tie ? 1 : 0;
                }
                cnt = w;
#pragma unroll
                for (int e = 0; e < kRoom; ++e)
                    if (((live >> e) & 1u) && score(e) == tau) {
                        if (ties <= 0) live &= ~(1u << e);
                        --ties;
                    }
            }
            to = pool_at + cnt * (8 * kTileTok);
            uint32_t at[kRoom];
#pragma unroll
            for (int e = 0; e < kRoom; ++e) {
                at[e] = to;
                to += ((live >> e) & 1u) * (8 * kTileTok);
            }
#pragma unroll
            for (int e = 0; e < kRoom; ++e)
                if ((live >> e) & 1u) st_entry(at[e], raw[e]);          // (the pool may be full)
            cnt = static_cast<int>(to - pool_at) / (8 * kTileTok);
        }
        tn += nsteps > 0 ? 1 : 0;
        // (after a timeout the thread still walks through the tile's barriers; every warp leaves together below)
        if (!ok) { set_status(a.status, kDevTimeout); *reinterpret_cast<volatile int*>(&sm.abort) = 1; }

        // Scores of -inf (chunks that the bias masks) and NaN beat no threshold, so fewer than K may have been kept: the lowest
        // of the other ids fill the places, as ties do.  With x the last of them, that makes every id up to x.
        const int miss = min(K, my_ncand) - cnt;
        if (ok && nsteps > 0 && tok < s.R && miss > 0) {
            int x = miss - 1, below = 0;
#pragma unroll 1
            while (below < cnt && static_cast<int>(pool[below * kTileTok] & 0xffffffffull) <= x) { ++below; ++x; }
#pragma unroll 1
            for (int e = cnt - 1; e >= below; --e) pool[(e + miss) * kTileTok] = pool[e * kTileTok];
#pragma unroll 1
            for (int e = 0; e <= x; ++e) pool[e * kTileTok] = static_cast<unsigned long long>(e);
            cnt += miss;
        }
        // the survivors are the selection, already in ascending chunk order; -1 padded
        int ids[N];
#pragma unroll
        for (int e = 0; e < N; ++e) ids[e] = nsteps == 0 ? (e < min(K, my_ncand) ? e : -1) : e < cnt ? static_cast<int>(pool[e * kTileTok] & 0xffffffffull) : -1;
        if (tok < s.R) {
            int32_t* sel = a.sel + (static_cast<long long>(pair) * s.R + tok) * K;
            if (((reinterpret_cast<uintptr_t>(sel) | static_cast<uintptr_t>(4 * K)) & 15) == 0) {     // rows of whole 16-byte pieces
#pragma unroll
                for (int e = 0; e < N; e += 4)
                    if (e < K) *reinterpret_cast<int4*>(sel + e) = make_int4(ids[e], ids[e + 1], ids[e + 2], ids[e + 3]);
            } else {
#pragma unroll
                for (int e = 0; e < N; ++e)
                    if (e < K) sel[e] = ids[e];
            }
        }
        if (a.cnt && ti * kTileTok >= a.t0) {
            // chunk histogram of this tile's entries (selected chunks + the chunks of each token's local window) in the
            // pools' shared memory (every thread holds its ids in registers by now), then one global add per used bin
            int* hist = reinterpret_cast<int*>(lists + 2 * kRoom * kTileTok);
            const bool in_smem = a.nc * sizeof(int) <= sizeof(unsigned long long) * kMaxK * kTileTok;
            int* gcnt = a.cnt + (static_cast<long long>((ti * kTileTok - a.t0) / a.qb) * pairs + pair) * a.nc;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (in_smem) {
                for (int x = row; x < a.nc; x += kTileTok) hist[x] = 0;
                asm volatile("bar.sync 1, 128;" ::: "memory");
            }
            if (tok < s.R) {
                int* dst = in_smem ? hist : gcnt;
#pragma unroll
                for (int e = 0; e < N; ++e)
                    if (ids[e] >= 0) atomicAdd(dst + ids[e], 1);
                const int pos = s.pos0 + tok;
                if (a.local)
                    for (int c = local_lo(pos, s.W, kS) / kS; c <= pos / kS; ++c) atomicAdd(dst + c, 1);
            }
            if (in_smem) {
                asm volatile("bar.sync 1, 128;" ::: "memory");
                for (int x = row; x < a.nc; x += kTileTok)
                    if (hist[x]) atomicAdd(gcnt + x, hist[x]);
            }
        }
        // the pools' memory (histogram) is free for the next tile; after a timeout every warp leaves here
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (*reinterpret_cast<volatile int*>(&sm.abort)) break;
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == kMmaWarp) tmem_dealloc(tmem_base, kTmemCols);
}

}  // namespace

bool prefill_select_tc_supports(const Shape& s) {
    return s.K <= kMaxK && static_cast<long long>(s.B) * s.Hq * s.R < (1ll << 31);
}

int launch_prefill_select_tc(const Shape& s, const void* q, const void* landmarks, const float* bias, int32_t* sel,
                             int* status, int* cnt, int qb, int nc, int t0, int local_counted, cudaStream_t stream) {
    const int pairs = s.B * s.Hkv;
    CUtensorMap map_q, map_lm;
    if (!make_bf16_2d_map(&map_q, q, static_cast<uint64_t>(s.B) * s.Hq * s.R, kD, 64, kTileTok) ||
        !make_bf16_2d_map(&map_lm, landmarks, static_cast<uint64_t>(s.B) * s.Hl * s.C, kD, 64, kS))
        return HILS_ERR_CUDA;
    const size_t smem = kQBytes + kLmStages * kLmStageBytes + sizeof(unsigned long long) * 2 * kMaxK * kTileTok +
                        sizeof(TcSmem) + 1024;
    static PerDeviceOnce attr_once;
    if (attr_once.pending()) {
        if (cudaFuncSetAttribute(prefill_select_tc_kernel<16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(smem)) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_select_tc_kernel<32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(smem)) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_select_tc_kernel<16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(smem)) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_select_tc_kernel<32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(smem)) != cudaSuccess)
            return HILS_ERR_CUDA;
        attr_once.done();
    }
    TcArgs a{s, bias, sel, status, (cnt && qb % kTileTok == 0) ? cnt : nullptr, qb, nc, t0, local_counted};
    const int tiles = (s.R + kTileTok - 1) / kTileTok;
    const unsigned all_tiles = static_cast<unsigned>(pairs) * tiles;
    const unsigned nsm = static_cast<unsigned>(sm_count());
    const unsigned grid = all_tiles < nsm ? all_tiles : nsm;       // one persistent CTA per SM
    const bool perhead = s.Hl != s.Hkv;
    cudaError_t rc;
    if (s.K <= 16) {
        rc = launch_pdl(perhead ? prefill_select_tc_kernel<16, true> : prefill_select_tc_kernel<16, false>, dim3(grid), dim3(kThreads), smem, stream,
                        map_q, map_lm, a);
    } else {
        rc = launch_pdl(perhead ? prefill_select_tc_kernel<32, true> : prefill_select_tc_kernel<32, false>, dim3(grid), dim3(kThreads), smem, stream,
                        map_q, map_lm, a);
    }
    if (rc != cudaSuccess) return HILS_ERR_CUDA;
    return a.cnt ? 2 : 1;
}

}  // namespace hils
