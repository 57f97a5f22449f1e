// Tensor-core prefill kernels: bf16, d = 128, S = 64, G = 4, any local window of up to 16 chunks (W <= 897), one
// landmark per KV head or per query head (the latter with K <= 32: the tcgen05 selection kernel).
//
// With independent queries the tokens that select a chunk are scattered over the sequence, so the
// path is organised CHUNK-MAJOR: K/V of a chunk are staged once and reused by every query row that
// selected it; what moves per (token, chunk) pair is the query rows in and one bf16 output row out.
//
//   prefill_select  warp-MMA scoring + top-K, the fallback for K > 32 (the tcgen05 kernel lives in
//                   prefill_select_tc.cu): per (sequence, KV head, 64-token tile) it streams landmark tiles
//                   through a TMA ring, scores them for the 4 heads (Eq. surrogate top-k), takes the group
//                   max (App. C) and keeps an exact running top-K per token (ties: lower chunk id).
//   invert_*        turn sel_idx into per-(query block, pair, chunk) lists of (token, slot) entries, every list
//                   starting on a tile boundary, the table of attend tiles, and the (token, slot) -> entry map.
//   (prefill_attend_tc.cu: the tcgen05 attend kernel over that tile table; one normalised bf16 output row
//                   and the per-head chunk mass per entry, in entry order.)
//   prefill_fuse    per (token, KV head): the softmax over {surrogate scores} U {log Z_swa}
//                   (Eq. HiLS weights) that mixes the rows written by the attend kernel.
#include "internal.h"
#include "tma.cuh"

namespace hils {
namespace {

constexpr int kD = 128;
constexpr int kS = 64;
constexpr int kG = 4;
constexpr int kQBMin = 4096, kQBMax = 16384;  // tokens per pass of the invert/attend/fuse phases
constexpr int kQBLeast = 2048;               // (in a workspace that holds no more)
constexpr size_t kObufBytes = 5ull << 30;    // partial outputs that a call keeps at a time (at least those of kQBMin tokens)
constexpr int kSelStages = 3;
constexpr int kSelStageBytes = kS * kD * 2;  // 64 landmark rows

struct PArgs {
    Shape s;
    const __nv_bfloat16* q;
    const __nv_bfloat16* lm;
    const float* bias;
    __nv_bfloat16* out;
    float* lse;
    int32_t* sel;
    int* status;
    // scratch (per token block)
    int* cnt;               // [n_blocks*pairs*nc] rows of each (block, pair, chunk): selectors + own tokens
    int* cursor;            // [pairs*C]
    int* blk_toff;          // [n_blocks + 1] first tile of every query block (tiles are grouped by block)
    int* pair_toff;         // [n_blocks * pairs + 1] first tile of every (block, pair)
    int* seg_tiles;         // [ceil(lists / kSegLists)] tiles of each segment of lists
    int* off;               // [n_blocks*pairs*nc] first entry of each list; every list starts on a tile boundary
    int* entries;           // [max_tiles * tile_tok] (token_local << 8) | slot, grouped by (block, pair, chunk);
                            // slot K marks the token's own chunk (local branch); list tails up to the next tile
                            // boundary are padding
    int* epos;              // [pairs*L*(K+1)] entry index of every (token, slot), -1 = slot unused
    int4* tiles;            // [max_tiles] {pair, chunk, first entry, rows}
    __nv_bfloat16* obuf;    // [entries of one block][G][128] normalised per-chunk outputs, in entry order
    float* lam;             // [entries of one block][G] per-head surrogate scores; local slot: log Z_swa
    int t0;                 // first token of the chunk-major part (the ones before it go query-major)
    int i0, i1;             // token block [i0, i1) of the attend / fuse launch
    int blk;                // its index
    int n_blocks;           // query blocks of qb tokens
    int qb;                 // tokens per block the obuf / lam strides are sized for
    int nc;                 // chunk slots per pair in cnt/off/...: max(C, ceil(L / S))
    int tile_tok;           // entries per attend tile
    int max_tiles;
    int nl;                 // slots of a token's local window: max_local_slots(W), 0 where `out` and `lse` hold that branch
    int inv_parts, inv_tok; // parts of a query block's tokens that the inversion's CTAs take, tokens of a part
    int whole;              // obuf / lam cover all query blocks (indexed by global entry): one fuse launch per call
};

// ------------------------------------------------------------------------------------------ select
// Insert `key` into the unsorted K-entry list of one token (all 4 lanes of a quad call this with the
// same key).  tau / pmin track the smallest kept key (the K-th best so far) once the list is full.
__device__ __forceinline__ void quad_insert(unsigned long long* list, int K, int& cnt, unsigned long long& tau,
                                            int& pmin, unsigned long long key, int t, unsigned qmask) {
    if (cnt < K) {
        if (t == 0) list[cnt] = key;
        ++cnt;
        if (cnt < K) return;
    } else {
        if (t == 0) list[pmin] = key;
    }
    __syncwarp(qmask);
    unsigned long long mn = ~0ull;
    int pm = 0;
    for (int e = t; e < K; e += 4) {
        const unsigned long long x = list[e];
        if (x < mn) { mn = x; pm = e; }
    }
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        const unsigned long long om = __shfl_xor_sync(qmask, mn, o);
        const int op = __shfl_xor_sync(qmask, pm, o);
        if (om < mn) { mn = om; pm = op; }
    }
    tau = mn;
    pmin = pm;
    __syncwarp(qmask);
}

struct SelSmem {
    uint64_t full[kSelStages];
    uint64_t empty[kSelStages];
};

__global__ void __launch_bounds__(160, 1)
prefill_select_kernel(const __grid_constant__ CUtensorMap map_lm, const PArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    SelSmem& sm = *reinterpret_cast<SelSmem*>(ring + kSelStages * kSelStageBytes);
    unsigned long long* lists = reinterpret_cast<unsigned long long*>(ring + kSelStages * kSelStageBytes + 64);

    const Shape& s = a.s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pairs = s.B * s.Hkv;
    const int tiles_per_seq = (s.R + kS - 1) / kS;
    const int ci = tiles_per_seq - 1 - static_cast<int>(blockIdx.x) / pairs;      // heavy tiles first
    const int pair = static_cast<int>(blockIdx.x) % pairs;
    const int b = pair / s.Hkv, gk = pair % s.Hkv;
    // candidates of a token = the chunks left of its local window (Sec. 2.1); the tile's last token has the most
    const int ncand = local_lo(s.pos0 + min(s.R, (ci + 1) * kS) - 1, s.W, kS) / kS;
    const int nst = (ncand + kS - 1) / kS;
    const int K = s.K, Kp = K + 1;

    if (tid == 0) {
        for (int i = 0; i < kSelStages; ++i) { mbar_init(&sm.full[i], 1); mbar_init(&sm.empty[i], 4); }
        mbar_fence_init();
        tma_prefetch_desc(&map_lm);
    }
    __syncthreads();

    if (warp == 4) {
        if (lane == 0) {
            for (int it = 0; it < nst; ++it) {
                const int st = it % kSelStages;
                if (it >= kSelStages && !mbar_wait(&sm.empty[st], ((it / kSelStages) - 1) & 1)) {
                    set_status(a.status, kDevTimeout);
                    break;
                }
                uint8_t* dst = ring + st * kSelStageBytes;
                const int row = pair * s.C + it * kS;
                mbar_expect_tx(&sm.full[st], kSelStageBytes);
                tma_load_2d(dst, &map_lm, &sm.full[st], 0, row);
                tma_load_2d(dst + 8192, &map_lm, &sm.full[st], 64, row);
            }
        }
        return;
    }

    const int g = lane >> 2, t = lane & 3;
    const unsigned qmask = 0xfu << (lane & ~3);
    const int tokA = ci * kS + warp * 16 + g, tokB = tokA + 8;
    const int ldA = min(tokA, s.R - 1), ldB = min(tokB, s.R - 1);
    const int ncA = local_lo(s.pos0 + ldA, s.W, kS) / kS, ncB = local_lo(s.pos0 + ldB, s.W, kS) / kS;

    // A operands: this warp's 16 tokens, one fragment set per head of the group
    uint32_t aq[kG][8][4];
#pragma unroll
    for (int h = 0; h < kG; ++h) {
        const __nv_bfloat16* qh = a.q + (static_cast<long long>(b) * s.Hq + gk * kG + h) * s.R * kD;
        const __nv_bfloat16* ra = qh + static_cast<long long>(ldA) * kD;
        const __nv_bfloat16* rb = qh + static_cast<long long>(ldB) * kD;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            aq[h][ks][0] = *reinterpret_cast<const uint32_t*>(ra + ks * 16 + 2 * t);
            aq[h][ks][1] = *reinterpret_cast<const uint32_t*>(rb + ks * 16 + 2 * t);
            aq[h][ks][2] = *reinterpret_cast<const uint32_t*>(ra + ks * 16 + 8 + 2 * t);
            aq[h][ks][3] = *reinterpret_cast<const uint32_t*>(rb + ks * 16 + 8 + 2 * t);
        }
    }
    unsigned long long* listA = lists + static_cast<size_t>(warp * 16 + g) * Kp;
    unsigned long long* listB = lists + static_cast<size_t>(warp * 16 + g + 8) * Kp;
    int cntA = 0, cntB = 0, pminA = 0, pminB = 0;
    unsigned long long tauA = 0ull, tauB = 0ull;
    const float* bias = a.bias ? a.bias + static_cast<long long>(pair) * s.C : nullptr;
    bool dead = false;

    for (int it = 0; it < nst && !dead; ++it) {
        const int st = it % kSelStages;
        if (!mbar_wait(&sm.full[st], (it / kSelStages) & 1)) {
            if (lane == 0) set_status(a.status, kDevTimeout);
            dead = true;
            break;
        }
        const uint32_t lm_addr = smem_u32(ring + st * kSelStageBytes);
        const int c0 = it * kS;
        const int ntl = min(8, (ncand - c0 + 7) >> 3);
        for (int nt = 0; nt < ntl; ++nt) {
            uint32_t bf[8][2];
#pragma unroll
            for (int kp = 0; kp < 4; ++kp) {
                const int row = nt * 8 + (lane & 7);
                const int dim = kp * 32 + (lane >> 3) * 8;
                ldmatrix_x4(lm_addr + (dim >> 6) * 8192 + swz128(row, (dim & 63) >> 3), bf[2 * kp][0], bf[2 * kp][1],
                            bf[2 * kp + 1][0], bf[2 * kp + 1][1]);
            }
            float um[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int h = 0; h < kG; ++h) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) mma_bf16_16816(acc, aq[h][ks], bf[ks][0], bf[ks][1]);
#pragma unroll
                for (int v = 0; v < 4; ++v) um[v] = fmaxf(um[v], acc[v]);
            }
            // um[0..1]: token A, chunks cb, cb+1; um[2..3]: token B
            const int cb = c0 + nt * 8 + 2 * t;
            unsigned long long key[4];
            bool any = false;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int c = cb + (v & 1);
                const int nc_tok = v < 2 ? ncA : ncB;
                float u = um[v] * s.scale;
                if (bias && c < nc_tok) u += bias[c];
                key[v] = c < nc_tok ? select_key(u, c) : 0ull;
                any |= key[v] > ((v < 2) ? tauA : tauB);
            }
            if (__ballot_sync(kFullMask, any) == 0u) continue;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const bool pass = key[v] > ((v < 2) ? tauA : tauB);
                unsigned nib = (__ballot_sync(kFullMask, pass) >> (lane & ~3)) & 0xfu;
                while (nib) {
                    const int src = __ffs(nib) - 1;
                    nib &= nib - 1;
                    const unsigned long long x = __shfl_sync(qmask, key[v], (lane & ~3) + src);
                    if (v < 2) {
                        if (x > tauA) quad_insert(listA, K, cntA, tauA, pminA, x, t, qmask);
                    } else {
                        if (x > tauB) quad_insert(listB, K, cntB, tauB, pminB, x, t, qmask);
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.empty[st]);
    }

    // ascending chunk ids, -1 padded
    __syncwarp();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int tok = half == 0 ? tokA : tokB;
        const unsigned long long* list = half == 0 ? listA : listB;
        const int n = half == 0 ? cntA : cntB;
        if (tok >= s.R) continue;
        int32_t* sel = a.sel + ((static_cast<long long>(pair)) * s.R + tok) * K;
        for (int e = t; e < n; e += 4) {
            const int id = key_chunk(list[e]);
            int rank = 0;
            for (int j = 0; j < n; ++j) rank += key_chunk(list[j]) < id ? 1 : 0;
            sel[rank] = id;
        }
        for (int e = n + t; e < K; e += 4) sel[e] = -1;
    }
}

// ------------------------------------------------------------------------------------------ invert
// Slots of a token: 0..K-1 the selected chunks, K..K+nl-1 the chunks of its local window [l(i), i] (Sec. 2.1:
// l(i) is chunk-aligned, so the window is whole chunks plus the causal part of the token's own chunk).  Every
// local chunk is attended like a selected one, with its own softmax; its chunk mass is the exact log-sum-exp of
// its scores, so the softmax over all slots' masses reproduces the single softmax over the window (Eq. chunk mass).
__host__ __device__ inline int max_local_slots(int W) { return (W - 1 + kS - 1) / kS + 1; }
__device__ __forceinline__ int slot_chunk(const PArgs& a, int pair, int tok, int slot) {
    if (slot >= a.s.K) {
        const int pos = a.s.pos0 + tok;
        const int c = local_lo(pos, a.s.W, kS) / kS + (slot - a.s.K);
        return c <= pos / kS ? c : -1;
    }
    return a.sel[(static_cast<long long>(pair) * a.s.R + tok) * a.s.K + slot];
}

// Counting and filling go through shared memory: a CTA takes a range of one pair's tokens inside one query block, counts
// its entries per chunk there and adds each chunk's count to the global one at once.  (With an add in global memory per
// entry the long lists serialise: a chunk that every token of a block selects takes one add per token.)  Neighbouring
// lanes take neighbouring slots, so that selection and entry indexes are read and written in order and the lanes of a
// warp rarely meet at a counter.  More chunks than counters: the range is walked once per kInvCounters of them.
constexpr int kInvThreads = 512;
constexpr int kInvCounters = 8192;
constexpr int kInvBatch = 4;              // entries per thread whose loads are in flight together

struct InvPart {
    int pair, lo, hi, i0;                 // tokens [lo, hi) of the query block that starts at i0
    long long list0;                      // first list of (query block, pair)
};
__device__ __forceinline__ InvPart invert_part(const PArgs& a) {
    const int pairs = a.s.B * a.s.Hkv, x = static_cast<int>(blockIdx.x) / a.inv_parts;
    const int blk = x / pairs;
    InvPart p;
    p.pair = x % pairs;
    p.i0 = a.t0 + blk * a.qb;
    p.lo = p.i0 + static_cast<int>(blockIdx.x) % a.inv_parts * a.inv_tok;
    p.hi = min(min(p.lo + a.inv_tok, p.i0 + a.qb), a.s.R);
    p.list0 = static_cast<long long>(x) * a.nc;
    return p;
}
// f(token, slot, chunk or -1) for every (token, slot) of the part
template <class F>
__device__ __forceinline__ void invert_walk(const PArgs& a, const InvPart& p, F f) {
    const int K1 = a.s.K + a.nl;
    const int dt = kInvThreads / K1, ds = kInvThreads % K1;
    int tok = p.lo + static_cast<int>(threadIdx.x) / K1, slot = static_cast<int>(threadIdx.x) % K1;
    while (tok < p.hi) {
        int tk[kInvBatch], sl[kInvBatch], c[kInvBatch];
#pragma unroll
        for (int i = 0; i < kInvBatch; ++i) {
            tk[i] = tok;
            sl[i] = slot;
            c[i] = tok < p.hi ? slot_chunk(a, p.pair, tok, slot) : -1;
            tok += dt;
            slot += ds;
            if (slot >= K1) {
                slot -= K1;
                ++tok;
            }
        }
#pragma unroll
        for (int i = 0; i < kInvBatch; ++i)
            if (tk[i] < p.hi) f(tk[i], sl[i], c[i]);
    }
}
// counts of the chunks [c0, c0 + n) of the part
__device__ __forceinline__ void invert_histogram(const PArgs& a, const InvPart& p, int* ctr, int c0, int n) {
    for (int i = threadIdx.x; i < n; i += kInvThreads) ctr[i] = 0;
    __syncthreads();
    invert_walk(a, p, [&](int, int, int c) {
        if (c >= c0 && c - c0 < n) atomicAdd(&ctr[c - c0], 1);
    });
    __syncthreads();
}

__global__ void __launch_bounds__(kInvThreads, 3) invert_count_kernel(const PArgs a) {
    extern __shared__ int ctr[];
    pdl_wait();
    const InvPart p = invert_part(a);
    for (int c0 = 0; c0 < a.nc; c0 += kInvCounters) {
        const int n = min(kInvCounters, a.nc - c0);
        invert_histogram(a, p, ctr, c0, n);
        for (int i = threadIdx.x; i < n; i += kInvThreads)
            if (ctr[i] > 0) atomicAdd(&a.cnt[p.list0 + c0 + i], ctr[i]);
        __syncthreads();
    }
}

// Exclusive prefix sum of the tiles per list, ceil(cnt / tile_tok), in two launches of one CTA per kSegLists lists:
// segment sums first, then every CTA adds up the sums of the segments before its own and scans its segment.
// A list's first entry is its first tile x tile_tok, so the tiles of a query block cover one contiguous,
// tile-aligned range of entries.  (Small segments: the scan also writes the tile records, and 1024 lists can have 30,000 of
// them; 16K tokens, K = 16: inversion 48 -> 38 us with 256 lists and a warp per list.)
constexpr int kSegLists = 256;
__global__ void __launch_bounds__(kSegLists) invert_segsum_kernel(const PArgs a) {
    __shared__ int wsum[kSegLists / 32];
    pdl_wait();
    const int n = a.s.B * a.s.Hkv * a.nc * a.n_blocks;
    const int x = blockIdx.x * kSegLists + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int ct = x < n ? (a.cnt[x] + a.tile_tok - 1) / a.tile_tok : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ct += __shfl_xor_sync(kFullMask, ct, o);
    if (lane == 0) wsum[warp] = ct;
    __syncthreads();
    if (threadIdx.x == 0) {
        int v = 0;
        for (int w = 0; w < kSegLists / 32; ++w) v += wsum[w];
        a.seg_tiles[blockIdx.x] = v;
    }
}

__global__ void __launch_bounds__(kSegLists) invert_scan_kernel(const PArgs a) {
    __shared__ int wsum_t[kSegLists / 32];
    __shared__ int wpre[kSegLists / 32];
    pdl_wait();
    const Shape& s = a.s;
    const int per_blk = s.B * s.Hkv * a.nc;
    const int n = per_blk * a.n_blocks;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // tiles of all earlier segments
    int pre = 0;
    if (a.seg_tiles) {
        for (int sg = tid; sg < static_cast<int>(blockIdx.x); sg += kSegLists) pre += a.seg_tiles[sg];
    } else {
#pragma unroll 4
        for (int l = tid; l < static_cast<int>(blockIdx.x) * kSegLists; l += kSegLists) pre += (a.cnt[l] + a.tile_tok - 1) / a.tile_tok;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pre += __shfl_xor_sync(kFullMask, pre, o);
    if (lane == 0) wpre[warp] = pre;
    const int x = blockIdx.x * kSegLists + tid;
    const int ce = x < n ? a.cnt[x] : 0;
    const int ct = (ce + a.tile_tok - 1) / a.tile_tok;
    int it = ct;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int nt = __shfl_up_sync(kFullMask, it, o);
        if (lane >= o) it += nt;
    }
    if (lane == 31) wsum_t[warp] = it;
    __syncthreads();
    int bt = 0;
    for (int w = 0; w < kSegLists / 32; ++w) bt += wpre[w] + (w < warp ? wsum_t[w] : 0);
    const int ot = bt + it - ct, oe = ot * a.tile_tok;
    if (x < n) {
        a.off[x] = oe;
        if (x % per_blk == 0) a.blk_toff[x / per_blk] = ot;
        if (x % a.nc == 0) a.pair_toff[x / a.nc] = min(ot, a.max_tiles);
        if (x == n - 1) {
            a.blk_toff[a.n_blocks] = min(ot + ct, a.max_tiles);
            a.pair_toff[n / a.nc] = min(ot + ct, a.max_tiles);
        }
    }
    // the tile records, a list at a time
    for (int l = 0; l < 32; ++l) {
        const int lct = __shfl_sync(kFullMask, ct, l), lot = __shfl_sync(kFullMask, ot, l), lce = __shfl_sync(kFullMask, ce, l);
        const int lx = x - lane + l, pair = (lx % per_blk) / a.nc, c = lx % a.nc;
        for (int k = lane; k < lct; k += 32)
            if (lot + k < a.max_tiles)
                a.tiles[lot + k] = make_int4(pair, c, (lot + k) * a.tile_tok, min(a.tile_tok, lce - k * a.tile_tok));
    }
}

// The part's entries per chunk once more, room for them in each list, then a cursor per chunk in shared memory.
// Whole inversion, 16K tokens, K = 16, 8 KV heads, one query block: 204 -> 71 us; 128K tokens, K = 32, counts given:
// 694 -> 385 us, most of it the scattered 4-byte stores of the entries.
__global__ void __launch_bounds__(kInvThreads, 3) invert_fill_kernel(const PArgs a) {
    extern __shared__ int ctr[];
    pdl_wait();
    const InvPart p = invert_part(a);
    const int K1 = a.s.K + a.nl;
    int* epos = a.epos + static_cast<long long>(p.pair) * a.s.R * K1;
    for (int c0 = 0; c0 < a.nc; c0 += kInvCounters) {
        const int n = min(kInvCounters, a.nc - c0);
        invert_histogram(a, p, ctr, c0, n);
        for (int i = threadIdx.x; i < n; i += kInvThreads) {
            const long long list = p.list0 + c0 + i;
            if (ctr[i] > 0) ctr[i] = a.off[list] + atomicAdd(&a.cursor[list], ctr[i]);
        }
        __syncthreads();
        invert_walk(a, p, [&](int tok, int slot, int c) {
            int pos = -1;
            if (c >= c0 && c - c0 < n) {
                pos = atomicAdd(&ctr[c - c0], 1);
                if (pos < a.max_tiles * a.tile_tok) a.entries[pos] = ((tok - p.i0) << 8) | slot;
            } else if (c >= 0 || c0 > 0) {
                return;                   // another pass's chunk
            }
            epos[static_cast<long long>(tok) * K1 + slot] = pos;
        });
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------ routed scores
// With a separate routing query q-hat (Eq. Q-Cal) the chunk mass of a selected slot is scale * q-hat . k'_c + b'_c,
// not the q . k'_c that the attend kernel read off its score tile: this kernel overwrites those masses.  One CTA
// per tile, one warp per entry at a time; lane l covers dimensions 4l .. 4l+3.  Local slots keep their masses.
__global__ void __launch_bounds__(128) prefill_route_scores_kernel(const PArgs a) {
    pdl_wait();
    const Shape& s = a.s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t_begin = a.blk_toff[a.blk];
    const int tile = t_begin + static_cast<int>(blockIdx.x);
    if (tile >= a.blk_toff[a.blk + 1]) return;
    const int4 rec = a.tiles[tile];
    const int pair = rec.x, c = rec.y, first = rec.z, ntok = rec.w;
    if (c >= s.C) return;
    const int b = pair / s.Hkv, gk = pair % s.Hkv, per = s.Hl / s.Hkv;
    const int e0 = a.whole ? 0 : t_begin * a.tile_tok;
    for (int ei = warp; ei < ntok; ei += 4) {
        const int e = a.entries[first + ei];
        const int tok = a.i0 + (e >> 8), slot = e & 255;
        if (slot >= s.K) continue;
#pragma unroll
        for (int h = 0; h < kG; ++h) {
            const long long lrow = (static_cast<long long>(b) * s.Hl + gk * per + (per == 1 ? 0 : h)) * s.C + c;
            const uint2 qv = *reinterpret_cast<const uint2*>(a.q + ((static_cast<long long>(b) * s.Hq + gk * kG + h) * s.R + tok) * kD + lane * 4);
            const uint2 lv = *reinterpret_cast<const uint2*>(a.lm + lrow * kD + lane * 4);
            float dotp = __uint_as_float(qv.x << 16) * __uint_as_float(lv.x << 16);
            dotp = fmaf(__uint_as_float(qv.x & 0xffff0000u), __uint_as_float(lv.x & 0xffff0000u), dotp);
            dotp = fmaf(__uint_as_float(qv.y << 16), __uint_as_float(lv.y << 16), dotp);
            dotp = fmaf(__uint_as_float(qv.y & 0xffff0000u), __uint_as_float(lv.y & 0xffff0000u), dotp);
            dotp = warp_sum(dotp);
            if (lane == 0) a.lam[static_cast<long long>(first - e0 + ei) * kG + h] = dotp * s.scale + (a.bias ? a.bias[lrow] : 0.f);
        }
    }
}

// ------------------------------------------------------------------------------------------ fuse
// One warp per (sequence, KV head, token): softmax over {surrogate scores of the selected chunks} U
// {log Z_swa} per head (Eq. HiLS weights, inter-chunk factor) and the weighted sum of the rows that
// prefill_attend wrote.  The rows are found through the entry index of every (token, slot); an entry's
// 4 heads are 1 KB contiguous (two 16-byte loads per lane); lane l covers head l/16 (and head 2 + l/16),
// elements 8*(l%16)..+7.
constexpr int kFuseWarps = 4;
constexpr int kFuseRows = 96;             // rows mixed per token: K <= 64 selected + up to 16 local chunks, 3 x 32 lanes

// LOCAL_ROW: the local branch is one more row, in `out` and `lse` (a template parameter: its registers cost the other form
// resident warps).
template <bool LOCAL_ROW>
__global__ void __launch_bounds__(kFuseWarps * 32) prefill_fuse_kernel(const PArgs a) {
    __shared__ float wsm[kFuseWarps][kG][kFuseRows];
    __shared__ int esm[kFuseWarps][kFuseRows];
    pdl_wait();
    const Shape& s = a.s;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int K = s.K, K1 = K + a.nl, nblk = a.i1 - a.i0;
    const long long total = static_cast<long long>(s.B) * s.Hkv * nblk;
    const long long w = static_cast<long long>(blockIdx.x) * kFuseWarps + wib;
    if (w >= total) return;
    // (the pairs backwards: what the attend kernel wrote last is still in L2; 16K tokens 303 -> 299 us, a 2048-token slice 100 -> 97)
    const int pair = s.B * s.Hkv - 1 - static_cast<int>(static_cast<unsigned>(w) / static_cast<unsigned>(nblk));
    const int il = static_cast<int>(static_cast<unsigned>(w) % static_cast<unsigned>(nblk));
    const int b = pair / s.Hkv, gk = pair % s.Hkv;
    const int tok = a.i0 + il;
    // rows to mix: the selected chunks (slots 0..nsel-1), then the chunks of the local window (slots K..K+nl-1)
    const int pos = s.pos0 + tok;                    // sequence position of this query row
    const int lc = local_lo(pos, s.W, kS) / kS;      // first local chunk = number of candidate chunks
    const int nsel = min(K, lc);
    const int nl = LOCAL_ROW ? 0 : pos / kS - lc + 1;
    const int nrows = nsel + nl;
    const int e0 = a.whole ? 0 : a.blk_toff[a.blk] * a.tile_tok;   // first entry of this query block
    const int* ep = a.epos + (static_cast<long long>(pair) * s.R + tok) * K1;
    const float4* lam4 = reinterpret_cast<const float4*>(a.lam);
    float (*wv)[kFuseRows] = wsm[wib];
    int* ev = esm[wib];
    // entry (relative to the block) and the four heads' chunk masses of rows lane, lane + 32, lane + 64
    float lam[3][kG];
#pragma unroll
    for (int st = 0; st < 3; ++st) {
        const int r = lane + 32 * st;
        float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        if (r < nrows) {
            const int en = ep[r < nsel ? r : K + (r - nsel)] - e0;
            ev[r] = en;
            v = lam4[en];
        }
        lam[st][0] = v.x; lam[st][1] = v.y; lam[st][2] = v.z; lam[st][3] = v.w;
    }
    if (LOCAL_ROW && nrows == 0 && lane == 0) ev[0] = 0;          // (local branch alone: the loads below read a row that nobody uses)
    // (streaming loads: a partial row is read once.)  The first four rows are requested before the weights are worked out (their addresses need only the entries)
    __syncwarp();
    uint4 ra[4], rb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = max(min(u, nrows - 1), 0);
        const __nv_bfloat16* row = a.obuf + static_cast<long long>(ev[r]) * kG * kD;
        ra[u] = __ldcs(reinterpret_cast<const uint4*>(row + lane * 8));
        rb[u] = __ldcs(reinterpret_cast<const uint4*>(row + 256 + lane * 8));
    }
    const int hA = lane >> 4, hB = 2 + (lane >> 4), piece = lane & 15;
    const long long rowA = (static_cast<long long>(b) * s.Hq + gk * kG + hA) * s.R + tok;
    const long long rowB = (static_cast<long long>(b) * s.Hq + gk * kG + hB) * s.R + tok;
    // the local branch where the query-major kernel left it: one more row, in this token's rows of `out` and `lse`
    float lam_l[kG], w_l[kG] = {0.f, 0.f, 0.f, 0.f};
    uint4 la = make_uint4(0u, 0u, 0u, 0u), lb = la;
#pragma unroll
    for (int h = 0; h < kG; ++h) lam_l[h] = LOCAL_ROW ? a.lse[(static_cast<long long>(b) * s.Hq + gk * kG + h) * s.R + tok] : -INFINITY;
    if (LOCAL_ROW) {
        la = *reinterpret_cast<const uint4*>(a.out + rowA * kD + piece * 8);
        lb = *reinterpret_cast<const uint4*>(a.out + rowB * kD + piece * 8);
    }
    float lse_h = 0.f;
#pragma unroll
    for (int h = 0; h < kG; ++h) {
        float Mx = warp_max(fmaxf(fmaxf(lam[0][h], lam[1][h]), lam[2][h]));
        if (LOCAL_ROW) Mx = fmaxf(Mx, lam_l[h]);
        float ex[3];
#pragma unroll
        for (int st = 0; st < 3; ++st) ex[st] = __expf(lam[st][h] - Mx);
        const float ex_l = LOCAL_ROW ? __expf(lam_l[h] - Mx) : 0.f;
        const float D = warp_sum(ex[0] + ex[1] + ex[2]) + ex_l;
        const float inv = 1.f / D;
        w_l[h] = ex_l * inv;
#pragma unroll
        for (int st = 0; st < 3; ++st)
            if (lane + 32 * st < nrows) wv[h][lane + 32 * st] = ex[st] * inv;
        if (lane == h) lse_h = Mx + __logf(D);
    }
    __syncwarp();
    float accA[8], accB[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) { accA[x] = 0.f; accB[x] = 0.f; }
    auto fma8 = [](float (&acc)[8], const uint4& raw, float wgt) {
        const uint32_t wd[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            acc[2 * x] = fmaf(wgt, __uint_as_float(wd[x] << 16), acc[2 * x]);
            acc[2 * x + 1] = fmaf(wgt, __uint_as_float(wd[x] & 0xffff0000u), acc[2 * x + 1]);
        }
    };
    if (LOCAL_ROW) {
        fma8(accA, la, hA ? w_l[1] : w_l[0]);
        fma8(accB, lb, hA ? w_l[3] : w_l[2]);
    }
    // four rows at a time (8 loads in flight per lane)
    for (int r0 = 0; r0 < nrows; r0 += 4) {
        if (r0 > 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = min(r0 + u, nrows - 1);
                const __nv_bfloat16* row = a.obuf + static_cast<long long>(ev[r]) * kG * kD;
                ra[u] = __ldcs(reinterpret_cast<const uint4*>(row + lane * 8));
                rb[u] = __ldcs(reinterpret_cast<const uint4*>(row + 256 + lane * 8));
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (r0 + u < nrows) {
                fma8(accA, ra[u], wv[hA][r0 + u]);
                fma8(accB, rb[u], wv[hB][r0 + u]);
            }
        }
    }
    uint4 pa, pb;
    pa.x = pack_bf16(accA[0], accA[1]); pa.y = pack_bf16(accA[2], accA[3]);
    pa.z = pack_bf16(accA[4], accA[5]); pa.w = pack_bf16(accA[6], accA[7]);
    pb.x = pack_bf16(accB[0], accB[1]); pb.y = pack_bf16(accB[2], accB[3]);
    pb.z = pack_bf16(accB[4], accB[5]); pb.w = pack_bf16(accB[6], accB[7]);
    *reinterpret_cast<uint4*>(a.out + rowA * kD + piece * 8) = pa;
    *reinterpret_cast<uint4*>(a.out + rowB * kD + piece * 8) = pb;
    if (lane < kG) a.lse[(static_cast<long long>(b) * s.Hq + gk * kG + lane) * s.R + tok] = lse_h;
}

// HILS_FORCE_MMA_SELECT=1 keeps the warp-MMA selection kernel even where the tcgen05 one applies (used to
// cross-check the two implementations).
const bool g_force_mma_select = [] {
    const char* e = getenv("HILS_FORCE_MMA_SELECT");
    return e != nullptr && e[0] == '1';
}();
// HILS_PREFILL_QB overrides the query-block length (multiple of 64, for tuning runs); 0 = choose per call.
const int kQBEnv = [] {
    const char* e = getenv("HILS_PREFILL_QB");
    const int v = e ? atoi(e) : 0;
    return (v >= 64 && v % 64 == 0 && v <= (1 << 20)) ? v : 0;
}();
// Tokens per query block: the longer a block, the longer the lists of its chunks (fewer K/V loads and ragged last tiles), and
// the attend kernel's walk over one KV head at a time keeps the head's query rows in L2 (16 MB at 16384 tokens).  The
// partial outputs set the limit: attend + fuse at 16384 against 8192 and 4096 tokens, us:
// 32K tokens, K = 16: 1698, 1747, -;  64K tokens, K = 32: 6384, 6564, -;  16K tokens, K = 16: 763, 772, 811;  32768 gains nothing.
int pick_query_block(const Shape& s, int nl) {
    if (kQBEnv) return kQBEnv;
    const size_t per_tok = static_cast<size_t>(s.B) * s.Hkv * (s.K + nl) * kG * kD * sizeof(__nv_bfloat16);
    int qb = kQBMax;
    while (qb > kQBMin && qb * per_tok > kObufBytes) qb /= 2;
    return qb;
}
struct Plan {
    int qb, nc, n_blocks, max_tiles, max_blk_tiles, whole;
    size_t off_cnt, off_cursor, off_ntiles, off_ptiles, zero_bytes, off_seg, off_off, off_entries, off_epos, off_tiles, off_obuf, off_lam,
        total, obuf_tiles;
};

// (nl: slots of a token's local window, 0 where it goes query-major; qb_fixed: tokens per query block, 0 = the fastest;
// at_once: whether the partial outputs of all blocks may be kept)
Plan make_plan(const Shape& s, int qb_fixed, int t0, int nl, bool at_once = true) {
    Plan p;
    const int R = s.R - t0;                      // tokens of the chunk-major part
    const size_t pairs = static_cast<size_t>(s.B) * s.Hkv;
    const int QB = qb_fixed > 0 ? qb_fixed : pick_query_block(s, nl);
    const size_t blk = static_cast<size_t>(R < QB ? (R + 127) / 128 * 128 : QB);
    p.qb = static_cast<int>(blk);
    const size_t nchunks = (static_cast<size_t>(s.pos0) + s.R + kS - 1) / kS;     // chunks the queries can touch
    const size_t nc = static_cast<size_t>(s.C) > nchunks ? static_cast<size_t>(s.C) : nchunks;
    p.nc = static_cast<int>(nc);
    const size_t nblocks = (static_cast<size_t>(R) + blk - 1) / blk;
    p.n_blocks = static_cast<int>(nblocks);
    // tiles of a block <= its entries / tile + one ragged tile per list; a block's tokens see the chunks up to its end
    const size_t tt = static_cast<size_t>(attend_tc_tile_tokens());
    size_t all_tiles = 0, max_blk = 0;
    for (size_t b = 0; b < nblocks; ++b) {
        const size_t toks = (b + 1) * blk <= static_cast<size_t>(R) ? blk : static_cast<size_t>(R) - b * blk;
        const size_t vis = ((s.pos0 + t0 + b * blk + toks) + kS - 1) / kS;
        // (and never more than its entries: a list that exists holds at least one)
        const size_t ents = pairs * toks * (s.K + nl);
        const size_t ragged = pairs * (toks * (s.K + nl) / tt + (vis < nc ? vis : nc));
        const size_t tiles = (ents < ragged ? ents : ragged) + 1;
        all_tiles += tiles;
        max_blk = tiles > max_blk ? tiles : max_blk;
    }
    p.max_tiles = static_cast<int>(all_tiles);
    p.max_blk_tiles = static_cast<int>(max_blk);
    size_t off = 0;
    auto take = [&](size_t bytes, size_t align = 16) { size_t o = (off + align - 1) / align * align; off = o + bytes; return o; };
    p.off_cnt = take(sizeof(int) * nblocks * pairs * nc);
    p.off_cursor = take(sizeof(int) * nblocks * pairs * nc);
    p.off_ntiles = take(sizeof(int) * (nblocks + 1));
    p.zero_bytes = off;                         // cnt, cursor, blk_toff are cleared together once per call
    p.off_ptiles = take(sizeof(int) * (nblocks * pairs + 1));
    p.off_seg = take(sizeof(int) * ((nblocks * pairs * nc + kSegLists - 1) / kSegLists));
    p.off_off = take(sizeof(int) * nblocks * pairs * nc);
    p.off_entries = take(sizeof(int) * all_tiles * tt, 256);
    p.off_epos = take(sizeof(int) * pairs * s.R * (s.K + nl));
    p.off_tiles = take(sizeof(int4) * all_tiles);
    // Partial outputs of all query blocks at once where they fit: the fusion then runs as one launch
    // over the whole call instead of one per block (each launch pays its ramp and its last wave).
    p.whole = (at_once && nblocks > 1 && all_tiles * tt * kG * kD * sizeof(__nv_bfloat16) <= kObufBytes) ? 1 : 0;
    const size_t obuf_tiles = p.whole ? all_tiles : max_blk;
    p.obuf_tiles = obuf_tiles;
    p.off_obuf = take(sizeof(__nv_bfloat16) * obuf_tiles * tt * kG * kD, 256);
    p.off_lam = take(sizeof(float) * obuf_tiles * tt * kG);
    p.total = off;
    return p;
}
// The fastest plan that `bytes` of workspace hold (128K tokens, K = 32: 18.5 ms with the 5.3 GB of blocks of 16384 tokens, 19.4 with
// the 2.8 GB of 8192, 20.0 with 1.6 GB); the smallest one if none does.
Plan fitting_plan(const Shape& s, int t0, int nl, size_t bytes) {
    Plan least = make_plan(s, 0, t0, nl);
    if (least.total <= bytes) return least;
    for (int qb = kQBMax; qb >= kQBLeast; qb /= 2) {
        const Plan p = make_plan(s, qb, t0, nl, false);
        if (p.total <= bytes) return p;
        if (p.total < least.total) least = p;
    }
    return least;
}

}  // namespace

bool prefill_fast_supports(const Shape& s, int dtype) {
    // any window whose chunks fit the fuse kernel's row table; the warp-MMA selection fallback (K > 32) scores one
    // landmark row per KV head
    return dtype == HILS_BF16 && !s.is_decode && s.d == kD && s.S == kS && s.W >= 1 && max_local_slots(s.W) <= 16 &&
           (s.Hl == s.Hkv || (s.K <= 32 && prefill_select_tc_supports(s))) &&
           (s.Hl == s.Hkv || s.Hl == s.Hq) && s.G == kG &&
           s.K >= 1 && s.K <= 64 && static_cast<long long>(s.B) * s.Hkv * s.T < (1ll << 31) &&
           static_cast<long long>(s.B) * s.Hkv * s.C < (1ll << 24) &&
           static_cast<long long>(s.B) * s.Hkv * ((s.pos0 + s.R + kS - 1) / kS) < (1ll << 31) &&
           static_cast<long long>(s.B) * s.Hkv * s.R * (s.K + max_local_slots(s.W)) < (1ll << 31);
}

size_t prefill_fast_scratch_bytes(const Shape& s, bool least) {
    // (with a routing query nothing goes query-major; and fewer entries may take more scratch, where they just fit at once)
    const size_t bytes = least ? 0 : ~static_cast<size_t>(0);
    const int t0 = prefill_query_tokens(s), nl = max_local_slots(s.W);
    const size_t all = fitting_plan(s, 0, nl, bytes).total;
    const size_t rest = t0 < s.R ? fitting_plan(s, t0, prefill_local_query(s, t0) ? 0 : nl, bytes).total : 0;
    return all > rest ? all : rest;
}

// Parts of a query block that the inversion's CTAs take: some 8 CTAs per SM, none with fewer entries than its threads hold
// in one batch.  Returns the CTAs.
static unsigned invert_split(PArgs& a, const Plan& p) {
    const long long groups = static_cast<long long>(p.n_blocks) * a.s.B * a.s.Hkv;
    const int toks = a.s.R - a.t0 < a.qb ? a.s.R - a.t0 : a.qb, K1 = a.s.K + a.nl;
    const long long most = (static_cast<long long>(toks) * K1 + kInvThreads * kInvBatch - 1) / (kInvThreads * kInvBatch);
    const long long want = 8ll * sm_count() / groups;
    a.inv_parts = static_cast<int>(want < 1 ? 1 : want < most ? want : most);
    a.inv_tok = (toks + a.inv_parts - 1) / a.inv_parts;
    return static_cast<unsigned>(groups * a.inv_parts);
}
static size_t invert_smem(const PArgs& a) { return sizeof(int) * (a.nc < kInvCounters ? a.nc : kInvCounters); }

// The inverse index on its own (the backward pass walks the same chunk-major tiles): per-(query block, pair, chunk)
// entry lists and the tile table, built from a selection that is already in memory.
// (query blocks of 16384 tokens: of one KV head they take 33 MB of queries and output gradients and as much of fp32 dq,
// which L2 holds while the head is walked; and a chunk's list is long, so that its dk and dv are added up rarely)
constexpr int kQBIndex = 16384;
size_t inverse_index_bytes(const Shape& s) { return make_plan(s, kQBEnv ? kQBEnv : kQBIndex, 0, max_local_slots(s.W)).off_obuf; }

int build_inverse_index(const Shape& s, const int32_t* sel, void* scratch, size_t bytes, InverseIndex* ix,
                        cudaStream_t stream) {
    const Plan p = make_plan(s, kQBEnv ? kQBEnv : kQBIndex, 0, max_local_slots(s.W));
    if (bytes < p.off_obuf) return HILS_ERR_WORKSPACE;
    const int pairs = s.B * s.Hkv;
    char* sc = static_cast<char*>(scratch);
    PArgs a = {};
    a.s = s;
    a.sel = const_cast<int32_t*>(sel);
    a.cnt = reinterpret_cast<int*>(sc + p.off_cnt);
    a.cursor = reinterpret_cast<int*>(sc + p.off_cursor);
    a.blk_toff = reinterpret_cast<int*>(sc + p.off_ntiles);
    a.pair_toff = reinterpret_cast<int*>(sc + p.off_ptiles);
    a.n_blocks = p.n_blocks;
    a.seg_tiles = reinterpret_cast<int*>(sc + p.off_seg);
    a.off = reinterpret_cast<int*>(sc + p.off_off);
    a.entries = reinterpret_cast<int*>(sc + p.off_entries);
    a.epos = reinterpret_cast<int*>(sc + p.off_epos);
    a.tiles = reinterpret_cast<int4*>(sc + p.off_tiles);
    a.max_tiles = p.max_tiles;
    a.qb = p.qb;
    a.nc = p.nc;
    a.tile_tok = attend_tc_tile_tokens();
    a.nl = max_local_slots(s.W);
    if (cudaMemsetAsync(sc + p.off_cnt, 0, p.zero_bytes, stream) != cudaSuccess) return HILS_ERR_CUDA;
    const unsigned eb = invert_split(a, p);
    const unsigned nseg = static_cast<unsigned>((static_cast<long long>(p.n_blocks) * pairs * p.nc + kSegLists - 1) / kSegLists);
    if (launch_pdl(invert_count_kernel, dim3(eb), dim3(kInvThreads), invert_smem(a), stream, a) != cudaSuccess ||
        launch_pdl(invert_segsum_kernel, dim3(nseg), dim3(kSegLists), 0, stream, a) != cudaSuccess ||
        launch_pdl(invert_scan_kernel, dim3(nseg), dim3(kSegLists), 0, stream, a) != cudaSuccess ||
        launch_pdl(invert_fill_kernel, dim3(eb), dim3(kInvThreads), invert_smem(a), stream, a) != cudaSuccess)
        return HILS_ERR_CUDA;
    trace_mark("backward_invert", stream);
    ix->qb = p.qb;
    ix->nc = p.nc;
    ix->n_blocks = p.n_blocks;
    ix->max_tiles = p.max_tiles;
    ix->tile_tok = a.tile_tok;
    ix->entries = a.entries;
    ix->tiles = a.tiles;
    ix->blk_toff = a.blk_toff;
    ix->pair_toff = a.pair_toff;
    return 4;
}

int launch_prefill_fast(const Shape& s, const Tensors& t, cudaStream_t stream) {
    // the first n_qm tokens of every sequence see few chunks and go query-major (with q_route their mixing logits would not
    // be what that kernel's score tile holds)
    const int n_qm = t.q_route ? 0 : prefill_query_tokens(s);
    const int last_cand = local_lo(s.pos0 + s.R - 1, s.W, kS) / kS;
    if (n_qm == s.R && last_cand <= s.K) {
        // nothing to select either: one launch
        const int rc = launch_prefill_query_tc(s, t, 0, n_qm, 0, 1, stream);
        if (rc < 0) return rc;
        trace_mark("prefill_query", stream);
        return rc;
    }
    const int t0 = n_qm;
    const bool local_qm = !t.q_route && t0 < s.R && prefill_local_query(s, t0);
    const int nl = local_qm ? 0 : max_local_slots(s.W);
    const Plan p = fitting_plan(s, t0 < s.R ? t0 : 0, nl, t.scratch_bytes);
    if (t.scratch_bytes < p.total) return HILS_ERR_WORKSPACE;
    const int pairs = s.B * s.Hkv;
    char* sc = static_cast<char*>(t.scratch);
    PArgs a;
    a.s = s;
    // PArgs::q feeds the selection fallback and the routed-score kernel: the routing query (q itself unless given)
    a.q = static_cast<const __nv_bfloat16*>(t.q_route ? t.q_route : t.q);
    a.lm = static_cast<const __nv_bfloat16*>(t.landmarks);
    a.bias = t.bias;
    a.out = static_cast<__nv_bfloat16*>(t.out);
    a.lse = t.lse;
    a.sel = t.sel_idx;
    a.status = t.status;
    a.cnt = reinterpret_cast<int*>(sc + p.off_cnt);
    a.cursor = reinterpret_cast<int*>(sc + p.off_cursor);
    a.blk_toff = reinterpret_cast<int*>(sc + p.off_ntiles);
    a.pair_toff = reinterpret_cast<int*>(sc + p.off_ptiles);
    a.n_blocks = p.n_blocks;
    a.blk = 0;
    a.seg_tiles = reinterpret_cast<int*>(sc + p.off_seg);
    a.off = reinterpret_cast<int*>(sc + p.off_off);
    a.entries = reinterpret_cast<int*>(sc + p.off_entries);
    a.epos = reinterpret_cast<int*>(sc + p.off_epos);
    a.tiles = reinterpret_cast<int4*>(sc + p.off_tiles);
    a.obuf = reinterpret_cast<__nv_bfloat16*>(sc + p.off_obuf);
    a.lam = reinterpret_cast<float*>(sc + p.off_lam);
    a.max_tiles = p.max_tiles;
    a.qb = p.qb;
    a.nc = p.nc;
    a.tile_tok = attend_tc_tile_tokens();
    a.t0 = t0;
    a.nl = nl;
    a.i0 = 0;
    a.i1 = 0;
    a.whole = p.whole;

    // K, V: boxes of 64 dims x 64 keys; partial outputs: boxes of 64 dims x 32 rows (one epilogue warp's rows)
    CUtensorMap map_k, map_v, map_lm, map_o;
    if (!make_kv_map(&map_k, t.k, pairs, s.T, s.pos0 + s.R, kD, 64, kS) || !make_kv_map(&map_v, t.v, pairs, s.T, s.pos0 + s.R, kD, 64, kS) ||
        !make_bf16_2d_map(&map_lm, t.landmarks, static_cast<uint64_t>(pairs) * s.C, kD, 64, kS) ||
        !make_bf16_2d_map(&map_o, a.obuf, static_cast<uint64_t>(p.obuf_tiles) * a.tile_tok * kG, kD, 64, 32))
        return HILS_ERR_CUDA;

    const size_t sel_smem = kSelStages * kSelStageBytes + 64 + sizeof(unsigned long long) * 64 * (s.K + 1) + 1024;
    static PerDeviceOnce attr_once;
    if (attr_once.pending()) {
        const size_t sel_max = kSelStages * kSelStageBytes + 64 + sizeof(unsigned long long) * 64 * 65 + 1024;
        if (cudaFuncSetAttribute(prefill_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(sel_max)) != cudaSuccess)
            return HILS_ERR_CUDA;
        attr_once.done();
    }

    int launches = 0;
    const int tiles_per_seq = (s.R + kS - 1) / kS;
    // counters of the inverse index start at zero; the tcgen05 selection kernel fills the per-chunk entry counts itself
    if (t0 < s.R && cudaMemsetAsync(sc + p.off_cnt, 0, p.zero_bytes, stream) != cudaSuccess) return HILS_ERR_CUDA;
    bool counted = false;
    if (prefill_select_tc_supports(s) && !g_force_mma_select) {
        const int rc = launch_prefill_select_tc(s, a.q, t.landmarks, t.bias, t.sel_idx, t.status, t0 < s.R ? a.cnt : nullptr, a.qb, a.nc, t0, !local_qm,
                                                stream);
        if (rc < 0) return rc;
        counted = rc == 2;
    } else {
        prefill_select_kernel<<<static_cast<unsigned>(pairs) * tiles_per_seq, 160, sel_smem, stream>>>(map_lm, a);
        if (cudaGetLastError() != cudaSuccess) return HILS_ERR_CUDA;
    }
    trace_mark("prefill_select", stream);
    ++launches;
    if (n_qm > 0) {
        const int rc = launch_prefill_query_tc(s, t, 0, n_qm, 0, 0, stream);
        if (rc < 0) return rc;
        trace_mark("prefill_query", stream);
        launches += rc;
        if (n_qm == s.R) return launches;
    }
    if (local_qm) {
        const int rc = launch_prefill_query_tc(s, t, t0, s.R, 1, 0, stream);
        if (rc < 0) return rc;
        trace_mark("prefill_local", stream);
        launches += rc;
    }

    // inverse index for every query block at once: per-(block, pair, chunk) lists of (token, slot) entries
    // and the table of attend tiles, grouped by block
    {
        const unsigned eb = invert_split(a, p);
        if (!counted) {
            invert_count_kernel<<<eb, kInvThreads, invert_smem(a), stream>>>(a);
            ++launches;
        }
        const unsigned nseg = static_cast<unsigned>((static_cast<long long>(p.n_blocks) * pairs * p.nc + kSegLists - 1) / kSegLists);
        // From here on every kernel of the call is launched so that its launch and prologue overlap the previous
        // kernel's tail; each of them waits for its predecessors' results before its first dependent access.  None
        // triggers its dependents early: CTAs of the next kernel parked beside a running attend kernel cost 5 %.
        // Few lists: the scan's CTAs add up the lists before their own themselves (8192 tokens, K = 16: 430 -> 427 us for the call, a slice of
        // 2048 tokens at 48K 323 -> 318; in 32 segments a CTA reads 8000 counts)
        if (nseg <= 32) {
            a.seg_tiles = nullptr;
        } else {
            if (launch_pdl(invert_segsum_kernel, dim3(nseg), dim3(kSegLists), 0, stream, a) != cudaSuccess) return HILS_ERR_CUDA;
            ++launches;
        }
        if (launch_pdl(invert_scan_kernel, dim3(nseg), dim3(kSegLists), 0, stream, a) != cudaSuccess ||
            launch_pdl(invert_fill_kernel, dim3(eb), dim3(kInvThreads), invert_smem(a), stream, a) != cudaSuccess)
            return HILS_ERR_CUDA;
        trace_mark("prefill_invert", stream);
        launches += 2;
    }
    for (int i0 = t0, blk = 0; i0 < s.R; i0 += a.qb, ++blk) {
        a.i0 = i0;
        a.i1 = s.R < i0 + a.qb ? s.R : i0 + a.qb;
        a.blk = blk;
        if (!a.whole || blk == 0) {
            // one launch per query block, or a single launch that walks all of them (whole-call output buffers)
            const CUtensorMap maps[3] = {map_k, map_v, map_o};
            // With many tiles per (block, pair) the launch walks the pairs one after the other: all CTAs then gather the
            // query rows of one KV head at a time, which L2 keeps.  With few tiles the additional ends of chunk runs cost more:
            // at 29 tiles per CTA and pair 1202 -> 1026 us, at 20 200 -> 191, at 4 102 -> 115.
            const bool by_pair = static_cast<long long>(a.qb) * (s.K + nl) >= 12ll * a.tile_tok * sm_count();
            const int rc = launch_prefill_attend_tc(s, t.q, maps, t.landmarks, t.bias, a.entries, a.tiles,
                                                    by_pair ? a.pair_toff + blk * pairs : a.blk_toff + blk, by_pair ? pairs : 1, a.lam,
                                                    t.status, a.i0, a.whole, a.whole ? p.n_blocks : 1, a.qb, stream);
            if (rc < 0) return rc;
            trace_mark("prefill_attend", stream);
            ++launches;
        }
        if (t.q_route) {
            const int ntl = (p.max_blk_tiles);
            if (launch_pdl(prefill_route_scores_kernel, dim3(static_cast<unsigned>(ntl)), dim3(128), 0, stream, a) != cudaSuccess)
                return HILS_ERR_CUDA;
            trace_mark("prefill_route_scores", stream);
            ++launches;
        }
        if (a.whole) {
            // one fusion launch after the last block's attend, over every token of the call
            if (a.i1 < s.R) continue;
            a.i0 = t0;
        }
        const long long fuse_warps = static_cast<long long>(pairs) * (a.i1 - a.i0);
        if (launch_pdl(a.nl == 0 ? prefill_fuse_kernel<true> : prefill_fuse_kernel<false>, dim3(static_cast<unsigned>((fuse_warps + kFuseWarps - 1) / kFuseWarps)),
                       dim3(kFuseWarps * 32), 0, stream, a) != cudaSuccess)
            return HILS_ERR_CUDA;
        trace_mark("prefill_fuse", stream);
        ++launches;
    }
    return launches;
}

}  // namespace hils
