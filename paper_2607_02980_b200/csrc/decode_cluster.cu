// Decode in one launch: bf16, d = 128, S = 64, at most 8 query heads per KV head, one landmark per KV head, any local
// window of up to 16 chunks, top_k up to 128.
//
// A UNIT is one (sequence, KV head) with up to four of the sequence's newest tokens (multi-token decode; one otherwise).
// A thread-block cluster works on a unit from the landmark scores to the output row, so that nothing of it travels
// through global memory and no launch sits between the steps:
//   score    tiles of 64 candidate chunks are dealt to the CTAs and their warps, which stream the landmark rows by TMA and
//            leave the group scores u_c = max_h s^h_c in shared memory (chunks in the MMA rows, heads in its columns);
//   select   exact top-K over the cluster (ties to the lower chunk id): every CTA finds a score that its share of K of its
//            candidates reach, the smallest of these scores leaves little more than K candidates over the cluster, and
//            every CTA ranks those against each other (distributed shared memory);
//   attend   the selected chunks and the chunks of the local window are dealt to the CTAs and their warps; every warp owns
//            one K and one V buffer, refills each as soon as it has read it, and waits for nobody: S^T = K q^T (keys in
//            the MMA rows, token x head columns), the chunk's own softmax, O^T += V^T P^T.  The mixing logit of a
//            selected chunk comes from its landmark row, which travels with the K tile; the mix of Eq. (HiLS weights) is
//            a running maximum and two running sums per column, so that the order of the chunks does not matter;
//   combine  the warps' sums meet in shared memory, the CTAs' in distributed shared memory.
// Bound: HBM (landmarks scanned + selected K / V), and where a call has few units the chain of dependent steps.  One
// launch per step (decode_fast.cu) drains and ramps between short phases and leaves the memory idle during the
// selection.  Before / now, B200, us per call through the Python entry points, calls back to back: 1 x 6000 tokens, K = 16:
// 22.7 / 9.2; 8 x 4K-16K paged, K = 32, W = 512: 49.3 / 22.7; 64 x 64K, K = 32: 142.6 / 111 (6.2 TB/s); 4 x 1M, K = 64: 65.4 / 43.5;
// 16 x 8K-32K, four drafts, K = 32: 121 / 56.7.  Before this form of its short steps (landmark tiles asked for ahead of the queries, a
// tile's biases under its wait, items placed by rank with sel_idx sorted behind the loads, no integer division on the way) the same calls
// took 12.7, 28.2, 117.3, 46.8 and 62.2.  (The output's rounded division is 0.1 us of the first: without it means that lie half way between
// two bf16 numbers came out on the wrong side.)
// Draft tokens of one sequence retrieve mostly the same chunks: the union of their selections is loaded once, and all
// their heads fill the MMA's columns.
#include <stddef.h>

#include "internal.h"
#include "tma.cuh"

namespace hils {
namespace {

constexpr int kD = 128;
constexpr int kS = 64;
constexpr int kHalf = kS * kD * 2;                // a buffer: a chunk's K or V tile, or 64 landmark rows
constexpr int kLmRow = kD * 2;                    // the chunk's landmark row, beside the K buffer
constexpr int kMaxWarps = 6;
constexpr int kMaxK = 128;
constexpr int kMaxCluster = 16;
constexpr float kLog2e = 1.4426950408889634f;

struct CArgs {
    Shape s;
    const __nv_bfloat16* q;
    const __nv_bfloat16* q_route;
    const __nv_bfloat16* lm;
    const float* bias;
    const int32_t* seq_lens;
    const int32_t* block_table;
    int num_pages;
    __nv_bfloat16* out;
    float* lse;
    int32_t* sel;
    int* status;
    int cs, lcs;       // CTAs per cluster (a power of two), its logarithm
    int tg;            // tokens of a sequence per unit
    int lgp;           // logarithm of the columns per token: G rounded up to a power of two
    int list_cap;      // candidates per token a CTA can hold
    // byte offsets behind the buffers
    int off_items, off_ids;
};

// Distributed shared memory
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_peer(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float ld_peer_f(uint32_t a) { return __uint_as_float(ld_peer(a)); }
__device__ __forceinline__ int4 ld_peer4(uint32_t a) {
    int4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_peer_f(uint32_t a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
// (.aligned: the whole warp has to arrive at the instruction, so lanes that a branch before it took apart are brought together first)
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync(int cs) {
    if (cs > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
}

// Item of the attend phase: a chunk with, per token of the unit, the role it plays.
struct Item {
    int chunk;         // -1: nothing to do (a page id out of range)
    int row;           // first row of the chunk in the K / V tensor maps
    uint32_t flags;    // bit m: in token m's local window; bit 8 + m: selected by token m; bit 16: has a landmark row
};

// Candidates per token up to which every CTA scores and ranks all of them, without a histogram and without waiting for the others:
// about one per thread.  Us per call, by histogram / this way: 6K tokens (93 candidates) 11.8 / 9.3, 12K (190) 11.9 / 11.0, 16K (249) 11.9 /
// 14.1; clusters of one CTA 8K (124) 20.0 / 19.0, 12K 20.2 / 20.5; three warps 6K 50.6 / 48.5, 8K 50.8 / 51.4; four drafts 4K (63) 32.9 / 31.9,
// 8K 35.2 / 38.0.
__host__ __device__ inline int rank_all_most(bool multi, int warps, int cs) { return multi ? 64 : warps == 3 ? 96 : cs > 1 ? 192 : 128; }

template <int TG>
struct CSmem {
    static constexpr int kBins = TG == 1 ? 512 : 256;
    static constexpr int kCand = TG == 1 ? 256 : 128;      // candidates of a token that can be ranked against each other
    unsigned kmin, kmax;                       // span of this CTA's scores (ordered keys)
    float edge[TG];                            // published: score that this CTA's share of K of its candidates reach
    unsigned long long thr[TG];                // candidates from this key on are collected
    int cnt[TG];                               // this CTA's candidates collected
    int start[TG][kMaxCluster + 1];            // positions of the CTAs' candidates in `all`
    int len[TG], nc[TG];                       // tokens visible to the unit's token m, its candidate chunks
    int bad;                                   // tokens whose candidates do not fit (bit m)
    unsigned long long prefix;
    int remaining;
    float col_max[kMaxWarps][16], col_den[kMaxWarps][16];   // the warps' running maximum and denominator per column
    int wsum[kMaxWarps];
    uint64_t full[kMaxWarps][2];
    alignas(16) unsigned long long all[TG][kCand];         // the cluster's candidates (score key, ~chunk id)
    unsigned long long own[TG][kCand];         // this CTA's
    int hist[TG][kBins];                       // (last, with the scores behind it: see Shares)
};

// Where the CTAs of a cluster leave their shares of the quarter columns (32 dimensions) that this CTA writes, kRows of them, with
// their maxima and denominators.  They arrive while this CTA may still be at work, so they lie in what nobody has used since the
// last cluster barrier, the histogram and the scores behind it, and take no room from the lists (a group of four tokens with lists of
// 1000 candidates, or 5900 candidates of one, fill a CTA): the scores have been read by the barrier that published the counts.  Where every CTA
// ranks all candidates the last barrier is the first one, and their scores, which are few, lie behind the shares.
template <int TG>
struct Shares {
    static constexpr int kRows = TG == 1 ? 32 : 64;
    static constexpr int kBehind = kRows * (32 * 4 + 8) - static_cast<int>(sizeof(CSmem<TG>::hist));       // bytes of them behind the histogram
    static_assert(offsetof(CSmem<TG>, hist) + sizeof(CSmem<TG>::hist) == sizeof(CSmem<TG>) && sizeof(CSmem<TG>) % 16 == 0 && kBehind % 16 == 0,
                  "the scores follow the histogram");
    float row[kRows][32];
    float2 md[kRows];
};

// NT: MMA column tiles of 8 (token x head columns), TG: tokens per unit at most.
template <int NT, int TG>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
decode_cluster_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                      const __grid_constant__ CUtensorMap map_lm, const CArgs a) {
    using Sm = CSmem<TG>;
    constexpr int kBins = Sm::kBins;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* bufs = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const Shape& s = a.s;
    const int NW = blockDim.x >> 5, NTH = blockDim.x;
    const int CS = a.cs, K = s.K, G = s.G, Gp = 1 << a.lgp;
    uint8_t* tail = bufs + NW * (2 * kHalf) + NW * kLmRow;
    Sm& sm = *reinterpret_cast<Sm*>(tail);
    Item* items = reinterpret_cast<Item*>(tail + a.off_items);
    int* sel_ids = reinterpret_cast<int*>(tail + a.off_ids);                 // [TG][K] the selection, best first
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    uint8_t* kbuf = bufs + warp * (2 * kHalf);                               // this warp's buffers
    uint8_t* vbuf = kbuf + kHalf;
    uint8_t* lmrow = bufs + NW * (2 * kHalf) + warp * kLmRow;
    const int unit = blockIdx.x >> a.lcs, rank = blockIdx.x & (CS - 1);
    // quotient by the number of warps (3 or 6) of a number below 98304: the kernel is a chain of short steps, and a division takes as
    // long as some of them (quotients by CS and by the columns of a token are shifts)
    auto per_warp = [&](int n) { return static_cast<int>((static_cast<unsigned>(n) * 43691u) >> (NW == 3 ? 17 : 18)); };
    const int kvh = unit % s.Hkv;
    const int ngrp = (s.qps + a.tg - 1) / a.tg;
    const int seq = unit / s.Hkv / ngrp, tok0 = (unit / s.Hkv % ngrp) * a.tg;
    const int ntok = min(a.tg, s.qps - tok0);
    const int query0 = seq * s.qps + tok0;

    if (lane == 0) {                             // (a warp's barriers are its own: it may ask for its first tile before the others are here)
        mbar_init(&sm.full[warp][0], 1);
        mbar_init(&sm.full[warp][1], 1);
        mbar_fence_init();
        fence_proxy_async_smem();
    }
    if (tid == 0) {
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
        tma_prefetch_desc(&map_lm);
    }
    for (int x = tid; x < TG * kBins; x += NTH) sm.hist[x >> (TG == 1 ? 9 : 8)][x & (kBins - 1)] = 0;
    if (CS > 1) cluster_arrive();                // (waited for below: the others are there, and their histograms clear)
    pdl_wait();
    pdl_launch_dependents();

    // the unit's tokens: visible length, candidates, local window (Sec. 2.1)
    const int cache_len = a.seq_lens[seq];
    auto token_len = [&](int m) {                // 0: invalid (reported, empty outputs)
        const int n = m < ntok ? cache_len - (s.qps - 1) + tok0 + m : 0;
        return n < 1 || n > s.T ? 0 : n;
    };
    int nc_max = 0, lc_min = 0x7fffffff, len_max = 0;
#pragma unroll 1
    for (int m = 0; m < TG; ++m) {
        const int n = token_len(m), nc = n > 0 ? local_lo(n - 1, s.W, kS) / kS : 0;
        if (tid == 0) {
            sm.len[m] = n;
            sm.nc[m] = nc;
            sm.cnt[m] = 0;
            if (n == 0 && m < ntok && rank == 0) set_status(a.status, kDevBadIndex);
        }
        if (n > 0) { lc_min = min(lc_min, nc); nc_max = max(nc_max, nc); len_max = max(len_max, n); }
    }
    if (tid == 0) { sm.kmin = 0xffffffffu; sm.kmax = 0u; sm.bad = 0; }
    const bool any_list = nc_max > K;            // some token has more candidates than places
    const int ci_max = len_max > 0 ? (len_max - 1) / kS : -1;
    const int n_local = ci_max >= 0 ? ci_max - lc_min + 1 : 0;
    const float* bias = a.bias ? a.bias + (static_cast<long long>(seq) * s.Hl + kvh) * s.C : nullptr;

    // tiles of 64 candidates: tile n belongs to CTA n mod CS (its tile n / CS, of warp n / CS mod NW), so that every CTA
    // sees a sample of the whole sequence
    // (few candidates: every CTA scores and ranks all of them, and none waits for another)
    const bool rank_all = any_list && nc_max <= rank_all_most(TG > 1, NW, CS);
    const int lcs_t = rank_all ? 0 : a.lcs, rank_t = rank_all ? 0 : rank;
    const int n_tiles = any_list ? (((nc_max + 63) >> 6) - rank_t + (1 << lcs_t) - 1) >> lcs_t : 0;      // this CTA's
    const int my_tiles = n_tiles > warp ? per_warp(n_tiles - warp + NW - 1) : 0;
    const int cap = TG == 1 ? 0 : rank_all ? (nc_max + 63) & ~63 : a.list_cap;
    float* scores = reinterpret_cast<float*>(tail + sizeof(Sm) + (rank_all && CS > 1 ? Shares<TG>::kBehind : 0));      // [TG][cap]
    auto global_id = [&](int i) { return ((((i >> 6) << lcs_t) + rank_t) << 6) + (i & 63); };   // candidate of list position i
    const int lm_row0 = (seq * s.Hl + kvh) * s.C;

    // Buffers: the warp's lane 0 refills a buffer once the warp has read it.  Tiles alternate between the two; items put
    // K (and the landmark row) in the first, V in the second.
    auto fill_tile = [&](int i) {
        uint64_t* bar = &sm.full[warp][i & 1];
        uint8_t* dst = kbuf + (i & 1) * kHalf;
        const int row = lm_row0 + global_id((warp + i * NW) * 64);
        mbar_expect_tx(bar, kHalf);
        tma_load_2d(dst, &map_lm, bar, 0, row);
        tma_load_2d(dst + 8192, &map_lm, bar, 64, row);
    };
    // the first landmark tiles are asked for before everything that the scores need besides
    if (lane == 0) {
        if (my_tiles > 0) fill_tile(0);
        if (my_tiles > 1) fill_tile(1);
    }

    auto item_row = [&](int c) {
        if (c < 0 || c > ci_max) return -1;
        if (!a.block_table) return (seq * s.Hkv + kvh) * s.T + c * kS;
        const int page = a.block_table[static_cast<long long>(seq) * s.C + c];
        return page < 0 || page >= a.num_pages ? -1 : (page * s.Hkv + kvh) * kS;
    };
    // this CTA's share of the local chunks (item q of the unit goes to CTA q mod CS; the local chunks come first)
    const int my_local = n_local > rank ? (n_local - rank + CS - 1) >> a.lcs : 0;
    for (int j = tid; j < my_local; j += NTH) {
        const int c = lc_min + rank + j * CS, row = item_row(c);
        uint32_t f = c < nc_max ? 1u << 16 : 0u;
#pragma unroll 1
        for (int m = 0; m < ntok; ++m) {
            const int n = token_len(m);
            if (n > 0 && c >= local_lo(n - 1, s.W, kS) / kS && c <= (n - 1) / kS) f |= 1u << m;
        }
        if (row < 0) set_status(a.status, kDevBadIndex);
        items[j] = Item{row < 0 ? -1 : c, row, f};
    }

    // (one token) the rk-th best chunk becomes item n_local + rk of the unit
    auto place = [&](int rk, int c) {
        const int at = n_local + rk;
        if ((at & (CS - 1)) != rank) return;
        const int row = item_row(c);
        if (row < 0) set_status(a.status, kDevBadIndex);
        items[at >> a.lcs] = Item{row < 0 ? -1 : c, row, (1u << 8) | (1u << 16)};
    };

    // column n of the MMAs: token n / Gp, head n % Gp of the group; two words of the column's query per k-step
    auto col_row = [&](const __nv_bfloat16* src, int nt) -> const __nv_bfloat16* {
        const int col = nt * 8 + g, m = col >> a.lgp, h = col & (Gp - 1);
        if (m >= ntok || h >= G) return nullptr;
        return src + (static_cast<long long>(query0 + m) * s.Hq + kvh * G + h) * kD;
    };
    auto load_cols = [&](const __nv_bfloat16* src, uint32_t (&f)[8][NT][2]) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const __nv_bfloat16* row = col_row(src, nt);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                f[ks][nt][0] = row ? *reinterpret_cast<const uint32_t*>(row + ks * 16 + 2 * t) : 0u;
                f[ks][nt][1] = row ? *reinterpret_cast<const uint32_t*>(row + ks * 16 + 8 + 2 * t) : 0u;
            }
        }
    };
    uint32_t qf[8][NT][2];
    load_cols(a.q_route, qf);

    auto fill_k = [&](int i) {
        const Item it = items[warp + i * NW];
        uint64_t* bar = &sm.full[warp][0];
        if (it.chunk < 0) { mbar_arrive(bar); return; }
        const bool lm = (it.flags >> 16) & 1u;
        mbar_expect_tx(bar, kHalf + (lm ? kLmRow : 0));
        tma_load_2d(kbuf, &map_k, bar, 0, it.row);
        tma_load_2d(kbuf + 8192, &map_k, bar, 64, it.row);
        if (lm) bulk_load(lmrow, a.lm + static_cast<long long>(lm_row0 + it.chunk) * kD, kLmRow, bar);
    };
    auto fill_v = [&](int i) {
        const Item it = items[warp + i * NW];
        uint64_t* bar = &sm.full[warp][1];
        if (it.chunk < 0) { mbar_arrive(bar); return; }
        mbar_expect_tx(bar, kHalf);
        tma_load_2d(vbuf, &map_v, bar, 0, it.row);
        tma_load_2d(vbuf + 8192, &map_v, bar, 64, it.row);
    };
    bool ok = true;
    uint32_t uses0 = 0, uses1 = 0;                // times this warp has waited for each buffer
    auto wait_buf = [&](int which) {
        uint32_t& n = which ? uses1 : uses0;
        if (ok && !mbar_wait(&sm.full[warp][which], n & 1u)) {
            ok = false;
            if (lane == 0) set_status(a.status, kDevTimeout);
        }
        ++n;
    };
    const bool early = warp < my_local;           // the warp's first item is a local chunk: requested before the selection
    __syncthreads();
    if (lane == 0) {
        if (early && my_tiles == 0) fill_k(0);
        if (early && my_tiles <= 1) fill_v(0);
    }

    if (CS > 1) cluster_wait();

    // ------------------------------------------------------------------------------------------ score
    if (any_list) {
        float umin = INFINITY, umax = -INFINITY;
        for (int i = 0; i < my_tiles; ++i) {
            const int pos0 = (warp + i * NW) * 64, id0 = global_id(pos0);         // the tile's place in the list, its first candidate
            float bv[8];                               // (loaded under the wait: behind it, one after the other, they took 5000 cycles)
#pragma unroll
            for (int x = 0; x < 8; ++x) bv[x] = bias && id0 + x * 8 + g < nc_max ? bias[id0 + x * 8 + g] : 0.f;
            wait_buf(i & 1);
            const uint32_t tile = smem_u32(kbuf + (i & 1) * kHalf);
            float acc[4][NT][4];
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) acc[mt][nt][0] = acc[mt][nt][1] = acc[mt][nt][2] = acc[mt][nt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) {
                    const int row = mt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8, dim = ks * 16 + (lane >> 4) * 8;
                    uint32_t fr[4];
                    ldmatrix_x4(tile + (dim >> 6) * 8192 + swz128(row, (dim & 63) >> 3), fr[0], fr[1], fr[2], fr[3]);
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc[mt][nt], fr, qf[ks][nt][0], qf[ks][nt][1]);
                }
            __syncwarp();
            if (lane == 0) {
                if (i + 2 < my_tiles) fill_tile(i + 2);
                else if (early) { if (i & 1) fill_v(0); else fill_k(0); }
            }
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    const int r = mt * 16 + hr * 8 + g;
                    const bool live = id0 + r < nc_max;
                    const float bb = bv[mt * 2 + hr];
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        // heads of a token: columns m Gp .. m Gp + G - 1
                        const int h0 = (nt * 8 + 2 * t) & (Gp - 1);
                        const float s0 = acc[mt][nt][2 * hr] * s.scale + bb, s1 = acc[mt][nt][2 * hr + 1] * s.scale + bb;
                        auto put = [&](int m, float u, bool writer) {
                            if (m >= ntok || !writer || !live) return;
                            scores[m * cap + pos0 + r] = u;
                            umin = fminf(umin, u);
                            umax = fmaxf(umax, u);
                        };
                        if (Gp == 1) {
                            put(nt * 8 + 2 * t, s0, true);
                            put(nt * 8 + 2 * t + 1, s1, true);
                        } else {
                            float u = fmaxf(h0 < G ? s0 : -INFINITY, h0 + 1 < G ? s1 : -INFINITY);
                            if (Gp >= 4) u = fmaxf(u, __shfl_xor_sync(kFullMask, u, 1));
                            if (Gp >= 8) u = fmaxf(u, __shfl_xor_sync(kFullMask, u, 2));
                            put((nt * 8 + 2 * t) >> a.lgp, u, h0 == 0);
                        }
                    }
                }
        }
        if (!rank_all) {
            const unsigned lo = __reduce_min_sync(kFullMask, ordered_key(umin)), hi = __reduce_max_sync(kFullMask, ordered_key(umax));
            if (lane == 0) { atomicMin(&sm.kmin, lo); atomicMax(&sm.kmax, hi); }
        }

        // -------------------------------------------------------------------------------------- select
        // Each phase below runs once, so its instructions are mostly fetched cold: the loops are rolled and the tokens
        // share the code.  A token's list is walked by NW / ntok warps.
        const int n_list = n_tiles * 64;
        const int wpt = TG == 1 || ntok == 1 ? NW : NW == 3 ? 1 : ntok == 2 ? 3 : ntok == 3 ? 2 : 1;                     // max(1, NW / ntok)
        const int m_first = wpt == NW ? 0 : wpt == 1 ? warp : wpt == 2 ? warp >> 1 : warp >= 3;                          // warp / wpt
        const int m_step = wpt == NW ? 1 : wpt == 1 ? NW : wpt == 2 ? 3 : 2;                                             // NW / wpt
        const int li = (warp - m_first * wpt) * 32 + lane, ls = wpt * 32;
        if (rank_all) {
            __syncthreads();
            // the scores as ordered keys, padded to a multiple of four by the lowest one
#pragma unroll 1
            for (int m = m_first; m < ntok; m += m_step) {
                unsigned* keys = reinterpret_cast<unsigned*>(sm.all[m]);
                const int nc = sm.nc[m];
                for (int x = li; x < nc + 3; x += ls) keys[x] = x < nc ? ordered_key(scores[m * cap + x]) : 0u;
            }
        } else {
            __syncthreads();
            // A score that this CTA's share of K of its candidates reach, off a histogram with bins of equal width in the
            // score (the bins of a radix digit are equal in the exponent, and most scores share two or three exponents).
            // (both scaled by 2^-8: a mask of the lowest finite number spans more than 2^126, beyond which this division returns 0, and without
            // bins every candidate is collected and goes through the radix selection: 8 x 25,600 tokens, K = 16, 70 % masked 25.0 us, 20.4
            // with the bins)
            const float lo = key_to_float(sm.kmin), inv = __fdividef(kBins * 0x1p-8f, (key_to_float(sm.kmax) - lo) * 0x1p-8f);
            const bool cut = inv > 0.f && inv < INFINITY;              // (no span: every candidate is collected)
#pragma unroll 1
            for (int m = m_first; m < ntok; m += m_step) {
                if (sm.nc[m] <= K || !cut) continue;
                const int nc = sm.nc[m];
#pragma unroll 4
                for (int i = li; i < n_list; i += ls)
                    if (global_id(i) < nc)
                        atomicAdd(&sm.hist[m][min(kBins - 1, max(0, static_cast<int>((scores[m * cap + i] - lo) * inv)))], 1);
            }
            __syncthreads();
#pragma unroll 1
            for (int m = warp; m < ntok; m += NW) {
                // walk the bins from the top until the running count reaches `want` (all of them reach the lowest score)
                // This CTA's share of K: equal ones where each CTA holds a full tile of candidates.  Where there are fewer, those that
                // hold one share K (rounded up, plus one), and the others publish +inf: an empty CTA would leave no threshold, and
                // the best of a handful is a poor one (one sequence of 17K-29K tokens, 8 CTAs and 4-7 full tiles, K = 32: 28.2 us
                // by the radix selection below, 13.9 this way).
                const int full = sm.nc[m] >> 6;
                int want = (K + CS - 1) >> a.lcs;
                if (full < CS && K <= 64 * full) want = rank < full ? static_cast<int>(__fdividef(static_cast<float>(K), static_cast<float>(full))) + 1 : 0;
                constexpr int kPer = kBins / 32;
                const int* h = sm.hist[m] + kBins - kPer * (lane + 1);      // this lane's bins, the top one last
                int mine = 0;
#pragma unroll
                for (int x = 0; x < kPer; x += 4) {
                    const int4 v = *reinterpret_cast<const int4*>(h + x);
                    mine += v.x + v.y + v.z + v.w;
                }
                int inc = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int nn = __shfl_up_sync(kFullMask, inc, o);
                    if (lane >= o) inc += nn;
                }
                if (lane == 0) sm.edge[m] = want > 0 ? lo : INFINITY;
                __syncwarp();
                int cum = inc - mine;
                if (cum < want && inc >= want) {               // at most one lane
                    int x = kPer - 1;
                    while (x > 0 && (cum += h[x]) < want) --x;
                    const int b = kBins - kPer * (lane + 1) + x;
                    // (a little below the bin's edge: the bins were found by a rounded product)
                    if (b > 0) sm.edge[m] = lo + __fdividef(static_cast<float>(b) - 0.01f, inv);
                }
            }
            cluster_sync(CS);
            // the smallest edge of the cluster: at least K candidates reach it, and seldom many more
#pragma unroll 1
            for (int m = warp; m < ntok; m += NW) {
                float e = lane < CS ? ld_peer_f(peer_addr(smem_u32(&sm.edge[m]), lane)) : INFINITY;
                e = -warp_max(-e);
                if (lane == 0) sm.thr[m] = static_cast<unsigned long long>(ordered_key(e)) << 32;
            }
            __syncthreads();
            for (int pass = 0;; ++pass) {
#pragma unroll 1
                for (int m = m_first; m < ntok; m += m_step) {
                    const int nc = sm.nc[m];
                    if (nc <= K || (pass == 1 && !((sm.bad >> m) & 1))) continue;
                    const unsigned long long thr = sm.thr[m];
#pragma unroll 4
                    for (int i = li; i < n_list; i += ls) {
                        const int id = global_id(i);
                        const unsigned long long key = select_key(scores[m * cap + i], id);
                        if (id < nc && key >= thr) {
                            const int p = atomicAdd(&sm.cnt[m], 1);
                            if (p < Sm::kCand) sm.own[m][p] = key;
                        }
                    }
                }
                cluster_sync(CS);
#pragma unroll 1
                for (int m = warp; m < ntok; m += NW) {
                    int inc = lane < CS ? static_cast<int>(ld_peer(peer_addr(smem_u32(&sm.cnt[m]), lane))) : 0;
#pragma unroll
                    for (int o = 1; o < kMaxCluster; o <<= 1) {
                        const int nn = __shfl_up_sync(kFullMask, inc, o);
                        if (lane >= o) inc += nn;
                    }
                    if (lane < CS) sm.start[m][lane + 1] = inc;
                    if (lane == 0) sm.start[m][0] = 0;
                    if (lane == CS - 1 && sm.nc[m] > K && pass == 0 && (inc > Sm::kCand || inc < K)) atomicOr(&sm.bad, 1 << m);
                }
                __syncthreads();
                if (pass == 1 || sm.bad == 0) break;
                // Too many candidates at or above the edge (scores that agree in many chunks): the exact K-th best key
                // by radix selection over the cluster, eight bits at a time, score first, then the lower chunk id.
#pragma unroll 1
                for (int m = 0; m < ntok; ++m) {
                    if (!((sm.bad >> m) & 1)) continue;
                    unsigned long long prefix = 0ull, mask = 0ull;
                    int remaining = K;
#pragma unroll 1
                    for (int dgt = 0; dgt < 7; ++dgt) {
                        const int shift = dgt < 4 ? 56 - 8 * dgt : 48 - 8 * dgt;   // (chunk ids have 24 bits)
                        for (int x = tid; x < 256; x += NTH) sm.hist[m][x] = 0;
                        __syncthreads();
                        for (int i = tid; i < n_list; i += NTH) {
                            const int id = global_id(i);
                            const unsigned long long key = select_key(scores[m * cap + i], id);
                            if (id < sm.nc[m] && (key & mask) == prefix) atomicAdd(&sm.hist[m][(key >> shift) & 255u], 1);
                        }
                        cluster_sync(CS);
                        if (warp == 0) {
                            int h8[8], mine = 0;                        // bins 255 - 8 lane - x
#pragma unroll
                            for (int x = 0; x < 8; ++x) h8[x] = 0;
                            for (int r = 0; r < CS; ++r) {
                                const uint32_t src = peer_addr(smem_u32(&sm.hist[m][248 - 8 * lane]), r);
                                const int4 u = ld_peer4(src), v = ld_peer4(src + 16);
                                h8[7] += u.x; h8[6] += u.y; h8[5] += u.z; h8[4] += u.w;
                                h8[3] += v.x; h8[2] += v.y; h8[1] += v.z; h8[0] += v.w;
                            }
#pragma unroll
                            for (int x = 0; x < 8; ++x) mine += h8[x];
                            int inc = mine;
#pragma unroll
                            for (int o = 1; o < 32; o <<= 1) {
                                const int nn = __shfl_up_sync(kFullMask, inc, o);
                                if (lane >= o) inc += nn;
                            }
                            int cum = inc - mine;
                            if (cum < remaining && inc >= remaining) {      // one lane
#pragma unroll
                                for (int x = 0; x < 8; ++x) {
                                    if (cum < remaining && cum + h8[x] >= remaining) {
                                        sm.prefix = prefix | (static_cast<unsigned long long>(255 - 8 * lane - x) << shift);
                                        sm.remaining = remaining - cum;
                                    }
                                    cum += h8[x];
                                }
                            }
                        }
                        cluster_sync(CS);                               // (the histograms have been read)
                        prefix = sm.prefix;
                        remaining = sm.remaining;
                        mask |= 255ull << shift;
                    }
                    __syncthreads();
                    if (tid == 0) { sm.thr[m] = prefix | (255ull << 24); sm.cnt[m] = 0; }
                }
                __syncthreads();
            }
            // every CTA fetches all of them
#pragma unroll 1
            for (int m = m_first; m < ntok; m += m_step) {
                if (sm.nc[m] <= K) continue;
                const int n = min(sm.start[m][CS], Sm::kCand);
                for (int x = li; x < n; x += ls) {
                    int r = 0;
                    while (sm.start[m][r + 1] <= x) ++r;
                    const uint32_t src = peer_addr(smem_u32(&sm.own[m][x - sm.start[m][r]]), r);
                    const unsigned lo32 = ld_peer(src), hi32 = ld_peer(src + 4);
                    sm.all[m][x] = (static_cast<unsigned long long>(hi32) << 32) | lo32;
                }
            }
        }
        __syncthreads();
        // the K best by rank (their order does not matter to the attention; sel_idx is put in ascending order further down)
#pragma unroll 1
        for (int m = m_first; m < ntok; m += m_step) {
            if (sm.nc[m] <= K) continue;
            if (rank_all) {
                const uint4* keys = reinterpret_cast<const uint4*>(sm.all[m]);
                const int nc = sm.nc[m];
                for (int e = li; e < nc; e += ls) {
                    const unsigned mine = reinterpret_cast<const unsigned*>(keys)[e];
                    int rk = 0;                                      // (equal scores: the lower chunk first)
#pragma unroll 2
                    for (int f = 0; f < nc; f += 4) {
                        const uint4 k = keys[f >> 2];
                        rk += (k.x > mine || (k.x == mine && f < e)) + (k.y > mine || (k.y == mine && f + 1 < e)) +
                              (k.z > mine || (k.z == mine && f + 2 < e)) + (k.w > mine || (k.w == mine && f + 3 < e));
                    }
                    if (rk < K) {
                        sel_ids[m * K + rk] = e;
                        if (TG == 1) place(rk, e);
                    }
                }
                continue;
            }
            const int n = min(sm.start[m][CS], Sm::kCand);
            for (int e = li; e < n; e += ls) {
                const unsigned long long mine = sm.all[m][e];
                int rk = 0;
#pragma unroll 4
                for (int f = 0; f < n; ++f) rk += sm.all[m][f] > mine ? 1 : 0;
                if (rk < K) {
                    sel_ids[m * K + rk] = key_chunk(mine);
                    if (TG == 1) place(rk, key_chunk(mine));
                }
            }
        }
    }
    // a token with at most K candidates takes them all
#pragma unroll 1
    for (int m = 0; m < ntok; ++m)
        if (sm.nc[m] <= K)
            for (int e = tid; e < sm.nc[m]; e += NTH) {
                sel_ids[m * K + e] = e;
                if (TG == 1) place(e, e);
            }

    // ------------------------------------------------------------------------------------------ items
    int n_items = n_local + min(K, nc_max);
    if (TG > 1) {
        __syncthreads();
        // union of the tokens' selections in the order (token, rank); a chunk belongs to the first token that holds it
        auto holds = [&](int m, int c) {
            const int n = c < sm.nc[m] ? min(K, sm.nc[m]) : 0;
            int hit = 0;
#pragma unroll 8
            for (int j = 0; j < n; ++j) hit |= sel_ids[m * K + j] == c ? 1 : 0;
            return hit != 0;
        };
        int base = n_local;
        for (int x0 = 0; x0 < TG * K; x0 += NTH) {
            const int x = x0 + tid, m = x / K, e = x % K;
            bool mine = false;
            int c = 0;
            uint32_t f = 1u << 16;
            if (m < ntok && e < min(K, sm.nc[m])) {
                c = sel_ids[m * K + e];
                mine = c < lc_min;                                     // chunks of some token's window are local items
#pragma unroll 1
                for (int mm = 0; mm < ntok; ++mm)
                    if (holds(mm, c)) {
                        f |= 1u << (8 + mm);
                        if (mm < m) mine = false;
                    }
            }
            const unsigned vote = __ballot_sync(kFullMask, mine);
            if (lane == 0) sm.wsum[warp] = __popc(vote);
            __syncthreads();
            int at = base + __popc(vote & ((1u << lane) - 1u));
            for (int w = 0; w < NW; ++w) { if (w < warp) at += sm.wsum[w]; base += sm.wsum[w]; }
            if (mine && (at & (CS - 1)) == rank) {
                const int row = item_row(c);
                if (row < 0) set_status(a.status, kDevBadIndex);
                items[at >> a.lcs] = Item{row < 0 ? -1 : c, row, f};
            }
            if (x0 + NTH < TG * K) __syncthreads();
        }
        n_items = base;
        for (int j = tid; j < my_local; j += NTH) {
            const int c = items[j].chunk;
            if (c < 0) continue;
            uint32_t f = items[j].flags;
#pragma unroll 1
            for (int mm = 0; mm < ntok; ++mm)
                if (holds(mm, c)) f |= 1u << (8 + mm);
            items[j].flags = f;
        }
    }
    __syncthreads();
    const int cta_n = n_items > rank ? (n_items - rank + CS - 1) >> a.lcs : 0;
    const int my_n = cta_n > warp ? per_warp(cta_n - warp + NW - 1) : 0;           // this warp's items: warp, warp + NW, ...
    if (lane == 0 && my_n > 0 && !early) { fill_k(0); fill_v(0); }
    if (rank == 0) {
        // ascending chunk ids by rank, then -1
        for (int x = tid; x < ntok * K; x += NTH) {
            const int m = TG == 1 ? 0 : x / K, e = x - m * K, nc = sm.nc[m], n = min(K, nc);
            const int* ids = sel_ids + m * K;
            const int id = e < n ? ids[e] : -1;
            int pos = e;
            if (e < n && nc > K) {
                pos = 0;
#pragma unroll 8
                for (int j = 0; j < n; ++j) pos += ids[j] < id ? 1 : 0;
            }
            a.sel[(static_cast<long long>(query0 + m) * s.Hkv + kvh) * K + pos] = id;
        }
    }

    // ------------------------------------------------------------------------------------------ attend
    const bool routed = a.q != a.q_route;
    if (routed) load_cols(a.q, qf);
    const float sl2 = s.scale * kLog2e;
    float o[8][NT][4];
#pragma unroll
    for (int mt = 0; mt < 8; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) o[mt][nt][0] = o[mt][nt][1] = o[mt][nt][2] = o[mt][nt][3] = 0.f;
    float Mx[NT][2], Dn[NT][2];                   // this thread's columns: 8 nt + 2 t + {0, 1}
    int ctok[NT][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            Mx[nt][x] = kLowestLogit;
            Dn[nt][x] = 0.f;
            const int col = nt * 8 + 2 * t + x;
            ctok[nt][x] = (col & (Gp - 1)) < G ? col >> a.lgp : TG;           // token of the column (TG: none)
        }
    for (int i = 0; i < my_n; ++i) {
        const Item it = items[warp + i * NW];
        const float bb = bias && it.chunk >= 0 && ((it.flags >> 8) & 0xffu) != 0u ? bias[it.chunk] : 0.f;
        wait_buf(0);
        if (it.chunk < 0) {
            wait_buf(1);
            if (lane == 0 && i + 1 < my_n) { fill_k(i + 1); fill_v(i + 1); }
            continue;
        }
        const uint32_t k_addr = smem_u32(kbuf), v_addr = smem_u32(vbuf);
        const bool any_sel = ((it.flags >> 8) & 0xffu) != 0u, any_loc = (it.flags & 0xffu) != 0u;
        float sc[4][NT][4], lamp[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            lamp[nt][0] = lamp[nt][1] = lamp[nt][2] = lamp[nt][3] = 0.f;
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) sc[mt][nt][0] = sc[mt][nt][1] = sc[mt][nt][2] = sc[mt][nt][3] = 0.f;
        }
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                const int row = mt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8, dim = ks * 16 + (lane >> 4) * 8;
                uint32_t fr[4];
                ldmatrix_x4(k_addr + (dim >> 6) * 8192 + swz128(row, (dim & 63) >> 3), fr[0], fr[1], fr[2], fr[3]);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(sc[mt][nt], fr, qf[ks][nt][0], qf[ks][nt][1]);
            }
        if (any_sel) {
            // every row of this A tile is the landmark row: each thread receives its own columns' products
            const uint32_t l_addr = smem_u32(lmrow);
            float lam2[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) lam2[nt][0] = lam2[nt][1] = lam2[nt][2] = lam2[nt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                uint32_t fr[4];
                ldmatrix_x4(l_addr + (ks * 16 + (lane >> 4) * 8) * 2, fr[0], fr[1], fr[2], fr[3]);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    uint32_t b0 = qf[ks][nt][0], b1 = qf[ks][nt][1];
                    if (routed) {
                        const __nv_bfloat16* row = col_row(a.q_route, nt);
                        b0 = row ? *reinterpret_cast<const uint32_t*>(row + ks * 16 + 2 * t) : 0u;
                        b1 = row ? *reinterpret_cast<const uint32_t*>(row + ks * 16 + 8 + 2 * t) : 0u;
                    }
                    mma_bf16_16816(ks & 1 ? lam2[nt] : lamp[nt], fr, b0, b1);
                }
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) { lamp[nt][0] += lam2[nt][0]; lamp[nt][1] += lam2[nt][1]; }
        }
        __syncwarp();
        if (lane == 0 && i + 1 < my_n) fill_k(i + 1);
        float f_[NT][2];
        bool moved = false;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const int m = ctok[nt][x];
                const bool loc = m < TG && ((it.flags >> m) & 1u), sel = m < TG && ((it.flags >> (8 + m)) & 1u);
                if (any_loc) {
                    // last visible key of the column; in a column whose token does not see the chunk, the last one that exists
                    // (rows past the unit's last token may hold anything, and a NaN outlives the weight of 0)
                    const int lim = (loc ? sm.len[m] : len_max) - 1 - it.chunk * kS;
#pragma unroll
                    for (int mt = 0; mt < 4; ++mt) {
                        if (mt * 16 + g > lim) sc[mt][nt][x] = -INFINITY;
                        if (mt * 16 + 8 + g > lim) sc[mt][nt][2 + x] = -INFINITY;
                    }
                }
                float mx = fmax3(sc[0][nt][x], sc[0][nt][2 + x], sc[1][nt][x]);
                mx = fmax3(mx, sc[1][nt][2 + x], sc[2][nt][x]);
                mx = fmax3(mx, sc[2][nt][2 + x], sc[3][nt][x]);
                mx = fmaxf(mx, sc[3][nt][2 + x]);
                mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, 4));
                mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, 8));
                mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, 16));
                float z = 0.f;
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) {
                    sc[mt][nt][x] = ex2_approx((sc[mt][nt][x] - mx) * sl2);
                    sc[mt][nt][2 + x] = ex2_approx((sc[mt][nt][2 + x] - mx) * sl2);
                    z += sc[mt][nt][x] + sc[mt][nt][2 + x];
                }
                z += __shfl_xor_sync(kFullMask, z, 4);
                z += __shfl_xor_sync(kFullMask, z, 8);
                z += __shfl_xor_sync(kFullMask, z, 16);
                float pw = 0.f;
                f_[nt][x] = 1.f;
                if (loc || sel) {
                    const float lam = sel ? lamp[nt][x] * s.scale + bb : mx * s.scale + __logf(z);
                    const float nm = fmaxf(Mx[nt][x], lam);
                    f_[nt][x] = __expf(Mx[nt][x] - nm);
                    const float w = __expf(lam - nm);
                    Dn[nt][x] = fmaf(Dn[nt][x], f_[nt][x], w);
                    Mx[nt][x] = nm;
                    pw = quotient(w, z);
                }
                moved = moved || f_[nt][x] != 1.f;
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) { sc[mt][nt][x] *= pw; sc[mt][nt][2 + x] *= pw; }
            }
        if (__any_sync(kFullMask, moved)) {
#pragma unroll
            for (int mt = 0; mt < 8; ++mt)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    o[mt][nt][0] *= f_[nt][0]; o[mt][nt][1] *= f_[nt][1];
                    o[mt][nt][2] *= f_[nt][0]; o[mt][nt][3] *= f_[nt][1];
                }
        }
        // the probabilities become the B operand by 8 x 8 transpositions
        uint32_t pb[4][NT][2];
#pragma unroll
        for (int mt = 0; mt < 4; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                pb[mt][nt][0] = movmatrix_trans(pack_bf16(sc[mt][nt][0], sc[mt][nt][1]));
                pb[mt][nt][1] = movmatrix_trans(pack_bf16(sc[mt][nt][2], sc[mt][nt][3]));
            }
        wait_buf(1);
        const int n_valid = len_max - it.chunk * kS;
        if (n_valid < kS) {
            // rows past the unit's last token may hold anything: zero them before they meet probabilities of 0
            for (int x = lane; x < (kS - n_valid) * 16; x += 32) {
                const int row = n_valid + (x >> 4), piece = x & 15;
                *reinterpret_cast<uint4*>(vbuf + (piece >> 3) * 8192 + swz128(row, piece & 7)) = make_uint4(0u, 0u, 0u, 0u);
            }
            __syncwarp();
            fence_proxy_async_smem();             // (the buffer is overwritten by a bulk copy later)
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
                const int row = kk * 16 + (lane >> 4) * 8 + (lane & 7), dim = mt * 16 + ((lane >> 3) & 1) * 8;
                uint32_t fr[4];
                ldmatrix_x4_trans(v_addr + (dim >> 6) * 8192 + swz128(row, (dim & 63) >> 3), fr[0], fr[1], fr[2], fr[3]);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(o[mt][nt], fr, pb[kk][nt][0], pb[kk][nt][1]);
            }
        __syncwarp();
        if (lane == 0 && i + 1 < my_n) fill_v(i + 1);
    }

    // ------------------------------------------------------------------------------------------ combine
    constexpr int kRedRow = kD + 4;               // (padded: the four column pairs of a store miss each other's banks)
    // every warp leaves its sums in its own (drained) buffers: [column][kRedRow]
    {
        float* red = reinterpret_cast<float*>(kbuf);
#pragma unroll
        for (int mt = 0; mt < 8; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    float* dst = red + (nt * 8 + 2 * t + x) * kRedRow + mt * 16 + g;
                    dst[0] = o[mt][nt][x];
                    dst[8] = o[mt][nt][2 + x];
                }
        if (g == 0) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    sm.col_max[warp][nt * 8 + 2 * t + x] = Mx[nt][x];
                    sm.col_den[warp][nt * 8 + 2 * t + x] = Dn[nt][x];
                }
        }
    }
    __syncthreads();
    auto emit = [&](int cx, int dim, float v, float M, float den) {
        const int m = TG == 1 ? 0 : cx / G, h = cx - m * G;
        const bool live = sm.len[m] > 0;
        const long long orow = static_cast<long long>(query0 + m) * s.Hq + kvh * G + h;
        a.out[orow * kD + dim] = __float2bfloat16_rn(live ? v / den : 0.f);
        if (dim == 0) a.lse[orow] = live ? M + __logf(den) : 0.f;
    };
    // the warps' sums (fixed order: deterministic); a warp takes a column at a time
    Shares<TG>& shares = reinterpret_cast<Shares<TG>&>(sm.hist);
#pragma unroll 1
    for (int cx = warp; cx < ntok * G; cx += NW) {
        const int m = TG == 1 ? 0 : cx / G, col = m * Gp + cx - m * G;
        const float mw = lane < NW ? sm.col_max[lane][col] : -INFINITY;
        const float M = warp_max(mw), fw = mw == -INFINITY ? 0.f : __expf(mw - M);
        const float den = warp_sum(lane < NW ? sm.col_den[lane][col] * fw : 0.f);
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        const float* src = reinterpret_cast<const float*>(bufs) + col * kRedRow + lane;
#pragma unroll 1
        for (int w = 0; w < NW; ++w, src += 2 * kHalf / 4) {
            const float f = __shfl_sync(kFullMask, fw, w);
#pragma unroll
            for (int x = 0; x < 4; ++x) v[x] = fmaf(src[32 * x], f, v[x]);
        }
        __syncwarp();
        if (CS == 1) {
#pragma unroll
            for (int x = 0; x < 4; ++x) emit(cx, lane + 32 * x, v[x], M, den);
        } else {
            // a quarter of a column (32 dimensions) goes to the CTA that writes it
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const int qx = cx * 4 + x, at = (qx >> a.lcs << a.lcs) + rank;
                st_peer_f(peer_addr(smem_u32(&shares.row[at][lane]), qx & (CS - 1)), v[x]);
                if (lane < 2) st_peer_f(peer_addr(smem_u32(&shares.md[at]) + 4 * lane, qx & (CS - 1)), lane ? den : M);
            }
        }
    }
    if (CS == 1) return;
    cluster_sync(CS);
#pragma unroll 1
    for (int qx = warp * CS + rank; qx < ntok * G * 4; qx += NW * CS) {
        const int cx = qx >> 2, at = qx - rank;
        // lane r: CTA r's maximum and denominator
        const float2 md = lane < CS ? shares.md[at + lane] : make_float2(-INFINITY, 0.f);
        const float M = warp_max(md.x), f = md.x == -INFINITY ? 0.f : __expf(md.x - M), den = warp_sum(md.y * f);
        float n = 0.f;
#pragma unroll 2
        for (int r = 0; r < CS; ++r) n = fmaf(shares.row[at + r][lane], __shfl_sync(kFullMask, f, r), n);
        emit(cx, (qx & 3) * 32 + lane, n, M, den);
    }
}

template <int NT, int TG>
int set_attributes() {
    static PerDeviceOnce once;
    if (once.pending()) {
        if (cudaFuncSetAttribute(decode_cluster_kernel<NT, TG>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448) != cudaSuccess ||
            cudaFuncSetAttribute(decode_cluster_kernel<NT, TG>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return HILS_ERR_CUDA;
        once.done();
    }
    return HILS_OK;
}

template <int NT, int TG>
int launch(const CArgs& a, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& ml, int units, int warps,
           size_t smem, cudaStream_t stream) {
    if (set_attributes<NT, TG>() != HILS_OK) return HILS_ERR_CUDA;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(a.cs);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(units) * a.cs);
    cfg.blockDim = dim3(warps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = a.cs > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, decode_cluster_kernel<NT, TG>, mk, mv, ml, a) != cudaSuccess) return HILS_ERR_CUDA;
    trace_mark("decode_cluster", stream);
    return 1;
}

struct ClusterPlan {
    int cs, lcs, warps, tg, gp, nt, list_cap, off_items, off_ids, units;
    size_t smem;
};

// Clusters of 2^lcs CTAs that the device holds at once, one CTA of 6 warps (or two of 3) per SM; asked once per device.
// (Fewer than SMs / cluster size: a cluster stays inside a group of SMs whose number is no multiple of it.)
int resident_clusters(int per_sm, int lcs) {
    static int cached[64][2][5] = {};
    const int dev = PerDeviceOnce::device();
    if (dev >= 0 && cached[dev][per_sm - 1][lcs] > 0) return cached[dev][per_sm - 1][lcs];
    int n = sm_count() * per_sm >> lcs;
    if (lcs > 0) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1u << lcs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1u << lcs);
        cfg.blockDim = dim3(per_sm == 2 ? 96 : 192);
        cfg.dynamicSmemBytes = per_sm == 2 ? 115712 : 232448;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int got = 0;
        if (set_attributes<1, 1>() != HILS_OK ||
            cudaOccupancyMaxActiveClusters(&got, decode_cluster_kernel<1, 1>, &cfg) != cudaSuccess)
            return 0;
        n = got;
    }
    if (dev >= 0) cached[dev][per_sm - 1][lcs] = n;
    return n;
}

bool plan_tokens(const Shape& s, int tg, int n_sm, ClusterPlan* p) {
    p->gp = 1;
    while (p->gp < s.G) p->gp *= 2;
    p->tg = tg;
    const bool multi = tg > 1;
    p->nt = multi ? 2 : 1;
    const int TG = multi ? 4 : 1;
    const long long units = static_cast<long long>(s.B / s.qps) * s.Hkv * ((s.qps + tg - 1) / tg);
    if (units > (1 << 24)) return false;
    p->units = static_cast<int>(units);
    const int cand = (s.T - 1) / kS;
    const int local = (s.W - 1 + kS - 1) / kS + 1 + (multi ? 1 : 0);
    for (int step = 0; step < 2; ++step) {
        // all units at once with one CTA per SM (six warps: the selection's phases are short), else two
        const int per_sm = (units <= n_sm) == (step == 0) ? 1 : 2;
        p->warps = per_sm == 2 ? 3 : 6;
        // the smallest cluster that gives every warp at most one chunk and a dozen landmark tiles, as long as all units are
        // resident at once
        int lcs = 0;
        while ((2 << lcs) < kMaxCluster && ((p->warps << lcs) < s.K + local || (p->warps << lcs) * 12 * 64 < cand) &&
               units <= resident_clusters(per_sm, lcs + 1))
            ++lcs;
        const int cs = 1 << lcs;
        p->cs = cs;
        p->lcs = lcs;
        p->list_cap = ((cand + 63) / 64 + cs - 1) / cs * 64;
        // Long lists of units that take turns on the SMs.  Groups: apart, on three warps, is as fast or faster (20 x 51,200 tokens, four
        // drafts, us grouped / apart: 8 query heads per KV head 131 / 117, 4 heads 114 / 113; while all units are resident, 16 x 64K, 67 / 79).
        // Two CTAs per SM only where they do not add a turn (K = 16 - 32, us two / one: 32 x 108K tokens, 256 units, 48 / 52; 40 x 90K, 320
        // units, 88 / 85).
        const auto turns = [&](long long at_once) { return (units + at_once - 1) / at_once; };
        if (multi ? units > n_sm && p->list_cap > 768 : per_sm == 2 && p->list_cap > 1344 && 2 * turns(2 * n_sm) > turns(n_sm)) continue;
        size_t off = multi ? sizeof(CSmem<4>) : sizeof(CSmem<1>);
        auto take = [&](size_t bytes) { const size_t at = (off + 15) / 16 * 16; off = at + bytes; return static_cast<int>(at); };
        // the scores, or those of a short list that every CTA holds whole, behind the shares of the output
        const int most = rank_all_most(multi, p->warps, cs), whole = ((cand < most ? cand : most) + 63) / 64 * 64;
        const size_t list = sizeof(float) * TG * p->list_cap, shares = cs == 1 ? 0 : multi ? Shares<4>::kBehind : Shares<1>::kBehind;
        const size_t ranked = shares + sizeof(float) * TG * whole;
        take(list > ranked ? list : ranked);
        p->off_items = take(sizeof(Item) * ((TG * s.K + local + cs - 1) / cs + 1));
        p->off_ids = take(sizeof(int) * TG * s.K);
        p->smem = 1024 + off + static_cast<size_t>(p->warps) * (2 * kHalf + kLmRow);
        if (p->smem <= (per_sm == 2 ? 115712u : 232448u)) return true;
    }
    return false;
}

// Tokens per unit.  Sharing the loads of a sequence's draft tokens pays once the memory is what bounds the call; below
// that, a unit per token leaves shorter chains of dependent steps (measured, 4 tokens x 32K, us grouped / apart: 512
// (sequence, token, KV head) triples 67 / 76, 256 51 / 42, 128 38 / 25; with a window of nine chunks, which the tokens
// share whole, 160 triples 43 / 50).
bool plan_cluster(const Shape& s, int n_sm, ClusterPlan* p) {
    int gp = 1;
    while (gp < s.G) gp *= 2;
    int tg = s.qps < 16 / gp ? s.qps : 16 / gp;
    if (tg > 4) tg = 4;
    const long long apart = static_cast<long long>(s.B) * s.Hkv;
    if (apart <= n_sm || (apart <= 2 * n_sm && 8 * (s.W / kS) <= s.K)) tg = 1;
    return (tg > 1 && plan_tokens(s, tg, n_sm, p)) || plan_tokens(s, 1, n_sm, p);
}

}  // namespace

// Every decode shape with one landmark row per KV head and lists that fit, except few chunks from a short cache (top_k
// below 16 and at most 4096 tokens): callers rely on three kernels per call there (hils_last_launch_count), although one
// is faster too (K = 8, us three / one launch: 6000 tokens 21 / 12, 64 x 64K 89 / 59).
bool decode_cluster_supports(const Shape& s) {
    ClusterPlan p;
    return s.Hl == s.Hkv && (s.K >= 16 || s.T > 4096) && s.K <= kMaxK && plan_cluster(s, sm_count(), &p);
}

void decode_cluster_form(const Shape& s, int32_t* form) {
    ClusterPlan p;
    if (!decode_cluster_supports(s) || !plan_cluster(s, sm_count(), &p)) return;
    form[0] = p.tg;
    form[1] = p.warps;
    form[2] = p.cs;
    form[3] = rank_all_most(p.tg > 1, p.warps, p.cs);
}

int launch_decode_cluster(const Shape& s, const Tensors& t, cudaStream_t stream) {
    ClusterPlan p;
    if (!plan_cluster(s, sm_count(), &p)) return HILS_ERR_UNSUPPORTED;
    CArgs a;
    a.s = s;
    a.q = static_cast<const __nv_bfloat16*>(t.q);
    a.q_route = static_cast<const __nv_bfloat16*>(t.q_route ? t.q_route : t.q);
    a.lm = static_cast<const __nv_bfloat16*>(t.landmarks);
    a.bias = t.bias;
    a.seq_lens = t.seq_lens;
    a.block_table = t.block_table;
    a.num_pages = t.num_pages;
    a.out = static_cast<__nv_bfloat16*>(t.out);
    a.lse = t.lse;
    a.sel = t.sel_idx;
    a.status = t.status;
    a.cs = p.cs;
    a.lcs = p.lcs;
    a.tg = p.tg;
    a.lgp = 0;
    while ((1 << a.lgp) < p.gp) ++a.lgp;
    a.list_cap = p.list_cap;
    a.off_items = p.off_items;
    a.off_ids = p.off_ids;
    const int seqs = s.B / s.qps;
    CUtensorMap map_k, map_v, map_lm;
    const uint64_t rows = t.block_table ? static_cast<uint64_t>(t.num_pages) * s.Hkv * kS : static_cast<uint64_t>(seqs) * s.Hkv * s.T;
    if (!make_bf16_2d_map(&map_k, t.k, rows, kD, 64, kS) || !make_bf16_2d_map(&map_v, t.v, rows, kD, 64, kS) ||
        !make_bf16_2d_map(&map_lm, t.landmarks, static_cast<uint64_t>(seqs) * s.Hl * s.C, kD, 64, kS))
        return HILS_ERR_CUDA;
    return p.nt == 1 ? launch<1, 1>(a, map_k, map_v, map_lm, p.units, p.warps, p.smem, stream)
                     : launch<2, 4>(a, map_k, map_v, map_lm, p.units, p.warps, p.smem, stream);
}

}  // namespace hils
