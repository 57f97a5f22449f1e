// Backward of the HiLS operator on tcgen05 tensor cores (bf16, d = 128, S = 64, four query heads per KV head, one landmark
// per KV head), chunk-major: d K and d V of a chunk are accumulated in tensor memory over the queries that attend it.
// Formulas: backward.cu / the C header.
//
// A tile is 32 (token, slot) entries of the forward's inverse index x 4 heads = 128 rows against one 64-key chunk:
//   S = Q [K; k']^T (64 keys and, as key 64, the landmark: the row's surrogate score), T = dO V^T;
//   per row: the slot's softmax statistics, d S and W (the weights of the keys) to shared memory as bf16;
//   d Q = d S K; d K^T += Q^T d S and d V^T += dO^T W (both operands MN-major: the row tiles as they sit in shared memory).
// Warp roles of a persistent CTA: 0-3 and 4-7 two statistics groups (a row per thread, tiles alternate), 8-11 read-out,
// 12-15 gather of the Q and dO rows and d landmark, 16 loads K, V and landmark, 17 issues S and T, 18 the other products,
// 19 feeds the tile records and entries through a ring.
// Tensor memory: per tile parity 80 + 64 columns of S and T (at 0 and 240), 2 x 64 of d K^T and d V^T (384 ..), and d Q,
// which has 96 columns of its own (144 .. 239) and borrows the 32 of its tile's consumed S or T beside them.
// Bound: the read-out warps (93 % of the time busy).  d Q leaves as fp32 reductions, 64 KB per tile, for which L2 takes 2760 cycles
// whatever carries them (measured alone, 148 SMs: `red` in 128-byte runs, boxes of 512 B to 2 KB, bulk copies of rows).  A row per
// lane goes to shared memory swizzled and from there by tensor-map reductions, a box of 32 columns of an entry's four heads each: no
// second pass through registers, and no `red` in the queue of loads and stores that the gather needs.  Per piece of 32 columns a
// warp spends some 550 cycles until the rows are staged and 570 to issue eight boxes (a box costs its issuer 60 - 80 cycles; one
// issuing warp for all of them is slower, 3.2 ms for the pass, for half of them 2.10, and one staging buffer per warp 2.54).
// Backward pass of 16K tokens, K = 16, 32 heads, with its other kernels: 2.02 ms with rows turned through shared memory and added by
// `red`, 1.83 with the boxes; 1.52 without the reductions.
// The CTAs walk one (query block, KV head) after the other, so that its rows of q, dO and dq stay in L2.
// History of this kernel alone on that shape: 3.52 ms with one tile at a time between barriers; 2.56 ms with these roles and d Q
// written over its own S and T, whose slot is then held until the reductions have gone out; 2.38 ms with d Q in columns of
// its own; 2.00 ms with two thirds of the code; 1.65 ms before the boxes.
#include "internal.h"
#include "tma.cuh"

namespace hils {
namespace {

constexpr int kD = 128;
constexpr int kS = 64;
constexpr int kG = 4;
constexpr int kTok = 32;
constexpr int kRows = kTok * kG;
constexpr int kNS = 80;                         // score columns: 64 keys + landmark (+ 15 that nothing reads)
// Either K block (64 dims) of a chunk: 64 key rows, the landmark row, and 896 bytes that hold other things.  The score product
// reads them, and what follows the block, as key rows 65 .. 79: what comes out of that stays in columns of its own.
constexpr int kKBlock = 72 * 128, kKHole = 65 * 128;
constexpr int kKBytes = 2 * kKBlock;
constexpr int kVBytes = kS * kD * 2;
constexpr int kQBytes = kRows * kD * 2;
constexpr int kDsBytes = kRows * kS * 2;
constexpr int kStgBytes = 32 * 32 * 4;          // read-out of d Q: 32 rows x 32 columns of a warp, two buffers each
constexpr int kMeta = 4;                        // tiles whose records and entries are in shared memory at a time
constexpr int kTCol = 80, kDkCol = 384, kDvCol = 448;
__device__ __forceinline__ uint32_t slot_col(uint32_t par) { return par * 240u; }          // S of a tile of this parity (T: + kTCol)
__device__ __forceinline__ uint32_t dq_col(uint32_t par) { return par ? 144u : 112u; }     // its d Q
constexpr int kReadWarp = 8, kGatherWarp = 12, kLoadWarp = 16, kFrontWarp = 17, kBackWarp = 18;
constexpr int kThreads = 20 * 32;
constexpr float kLog2e = 1.4426950408889634f;
constexpr uint32_t kUmmaAMnMajor = 1u << 15;    // instruction-descriptor bit: A operand is MN-major

struct BArgs {
    Shape s;
    const __nv_bfloat16* q;
    const __nv_bfloat16* dout;
    const __nv_bfloat16* lm;
    const float* bias;
    const float* lse;
    const float* dsum;         // [B, Hq, R] dout . out
    const int* entries;
    const int4* tiles;
    const int* seg_toff;       // first tile of every segment (query block, or pair of one), n_seg + 1 entries
    int n_seg, segs, qb;       // segments, segments per query block, tokens per query block
    float* dq;
    float* dk;
    float* dv;
    float* dlm;
    float* dbias;
    int* status;
};

struct alignas(16) Tile {
    int ent[kTok];                              // (token of the query block) << 8 | slot
    int flags;                                  // entries (0: no more tiles) | first tile of its run << 8 | last << 9 | keys << 16
    int row0;                                   // q, dO, dq row of the query block's first token, head 0 of the KV head
    int kv;                                     // first k, v row of the chunk
    int lm;                                     // landmark row of the chunk (-1: none)
    int head0, tok0;                            // head 0 of the KV head (of all sequences'), the query block's first token
    int vis;                                    // last visible key of a local row: this + the token
};
struct BSmem {                                  // in the first K block's hole, behind d lambda
    uint64_t meta_full[kMeta], meta_empty[kMeta];
    uint64_t q_full[2];
    uint64_t k_ready, k_empty;
    uint64_t st_full[2], slot_empty[2];
    uint64_t ds_full[2], done[2];               // done: every product of the tile has completed
    uint64_t dq_full, dq_empty;
    uint64_t acc_empty;
    uint32_t tmem_base;
};
constexpr int kDlamBytes = kRows * 4;           // scale * d lambda of a tile's rows: in the hole of the K block of its parity
constexpr int kLmBytes = kD * 2;                // a run's landmark for the read-out: behind d lambda in the second hole, or last
static_assert(kKHole + kDlamBytes + sizeof(BSmem) <= kKBlock && kKHole + kDlamBytes + kLmBytes <= kKBlock, "what the holes hold");
constexpr size_t kSmemBytes = 4 * kQBytes + kKBytes + kVBytes + 2 * kDsBytes + 8 * kStgBytes + kMeta * sizeof(Tile) + kLmBytes;
static_assert(kSmemBytes <= 232448, "shared memory of the backward kernel");

__device__ __forceinline__ void red_add_f32(float* p, float x) {
    asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(x) : "memory");
}
// Adds one entry's box (32 columns x 1 token x 4 heads, 128B swizzle) to d Q; tracked by the issuing thread's bulk groups.
__device__ __forceinline__ void tma_red_add_3d(const CUtensorMap* map, const void* src, int x, int y, int z) {
    asm volatile("cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(map), "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void red_add_v4(float* p, float x, float y, float z, float w) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1)
backward_tc_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                   const __grid_constant__ CUtensorMap map_dq, const BArgs a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];     // (no room to round up: see tiles_aligned)
    uint8_t* qbuf = smem_raw;                    // [2]
    uint8_t* obuf = qbuf + 2 * kQBytes;          // dO rows [2]
    uint8_t* kbuf = obuf + 2 * kQBytes;
    uint8_t* vbuf = kbuf + kKBytes;
    uint8_t* dsbuf = vbuf + kVBytes;
    uint8_t* wbuf = dsbuf + kDsBytes;
    uint8_t* stgbuf = wbuf + kDsBytes;           // [4][2]
    Tile* const rec = reinterpret_cast<Tile*>(stgbuf + 8 * kStgBytes);
    BSmem& sm = *reinterpret_cast<BSmem*>(kbuf + kKHole + kDlamBytes);
    auto dlam_of = [&](uint32_t par) { return reinterpret_cast<float*>(kbuf + kKHole + par * kKBlock); };
    const Shape& s = a.s;
    const int tid = threadIdx.x, warp = __shfl_sync(kFullMask, tid >> 5, 0), lane = tid & 31;

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.q_full[i], 4 * 32 + 4);
            mbar_init(&sm.st_full[i], 1);
            mbar_init(&sm.slot_empty[i], 4);
            mbar_init(&sm.ds_full[i], 4);
            mbar_init(&sm.done[i], 1);
        }
        mbar_init(&sm.k_ready, 2);              // the TMA issuer's arrive.expect_tx + the landmark writer
        mbar_init(&sm.k_empty, 1);
        mbar_init(&sm.dq_full, 1);
        mbar_init(&sm.dq_empty, 4);
        mbar_init(&sm.acc_empty, 4);
        // (readers of a tile's record: four warps each of statistics, read-out and gather, and three threads)
        for (int i = 0; i < kMeta; ++i) { mbar_init(&sm.meta_full[i], 1); mbar_init(&sm.meta_empty[i], 15); }
        mbar_fence_init();
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
        tma_prefetch_desc(&map_dq);
    }
    if (warp == kFrontWarp) tmem_alloc(&sm.tmem_base, 512);
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(kFullMask, sm.tmem_base, 0);
    pdl_wait();

    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        if (ok && !mbar_wait(bar, parity)) ok = false;
        return ok;
    };
    // record of tile n of this CTA (false: there is none)
    auto tile_of = [&](uint32_t n) {
        if (!wait(&sm.meta_full[n % kMeta], (n / kMeta) & 1)) return false;
        return (rec[n % kMeta].flags & 255) != 0;
    };
    auto tile_done = [&](uint32_t n) { mbar_arrive(&sm.meta_empty[n % kMeta]); };       // one lane: this warp needs it no more
    const int hs = s.R;                          // rows between two heads of a token

    if (warp < kReadWarp) {
        // ================================================================ statistics: one row per thread
        const uint32_t grp = static_cast<uint32_t>(warp >> 2);
        const int row = (warp & 3) * 32 + lane, e_row = row >> 2, hd = row & 3;
        const uint32_t s_tm = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + slot_col(grp);
        const float c2 = s.scale * kLog2e;
        for (uint32_t n = grp; tile_of(n); n += 2) {
            const Tile& tl = rec[n % kMeta];
            const int n_ent = tl.flags & 255, ent = tl.ent[min(e_row, n_ent - 1)], lmr = tl.lm;
            const bool local = (ent & 255) >= s.K;
            // last visible key of the row; -1 for the rows of a ragged tile's padding
            const int limit = e_row >= n_ent ? -1 : local ? min(kS - 1, tl.vis + (ent >> 8)) : kS - 1;
            const int orow = tl.row0 + hd * hs + (ent >> 8);
            const float lse = __ldg(a.lse + orow), dsum = a.dsum[orow];
            const float bb = (a.bias && lmr >= 0) ? __ldg(a.bias + lmr) : 0.f;
            const bool masked = __any_sync(kFullMask, limit < kS - 1);
            if (lane == 0) tile_done(n);
            if (!wait(&sm.st_full[grp], (n >> 1) & 1)) break;
            tc_fence_after_sync();
            // The scores pass through three times and T twice, 16 columns of each at a time, the next piece's load under the
            // current one's arithmetic: kept in registers they would not fit beside 20 warps.  Rolled loops: the roles' code
            // together has to stay in the instruction cache (with less code for each role 16K tokens, K = 16 took 2.00 ms, not 2.38).
            uint32_t va[32], vb[32];
            if (masked) {
                // (rare) hide the keys past the row's last visible one
#pragma unroll 1
                for (int q = 0; q < 8; ++q) {
                    uint32_t w[8];
                    float x[4], y[4];
                    tmem_ld4(s_tm + 8 * q, x);
                    tmem_ld4(s_tm + 8 * q + 4, y);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        w[j] = __float_as_uint(8 * q + j <= limit ? x[j] : -INFINITY);
                        w[4 + j] = __float_as_uint(8 * q + 4 + j <= limit ? y[j] : -INFINITY);
                    }
                    tmem_st8(s_tm + 8 * q, w);
                }
                tmem_wait_st();
            }
            tmem_ld32_issue(s_tm, va);
            tmem_ld_wait32(va);
            tmem_ld32_issue(s_tm + 32, vb);
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            auto max32 = [&](const uint32_t (&v)[32]) {
#pragma unroll
                for (int j = 0; j < 32; j += 8)
#pragma unroll
                    for (int x = 0; x < 4; ++x) mx[x] = fmax3(mx[x], __uint_as_float(v[j + 2 * x]), __uint_as_float(v[j + 2 * x + 1]));
            };
            max32(va);
            tmem_ld_wait32(vb);
            tmem_ld16x2_issue(s_tm, s_tm + kTCol, va);
            max32(vb);
            float m = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            if (limit < 0) m = 0.f;
            // e_j = exp(x_j - m), their sum Z and sum e_j t_j
            const float2 c22 = make_float2(c2, c2), nm2 = make_float2(-m * c2, -m * c2);
            auto exp2_of = [&](const uint32_t (&v)[32], int j) {
                const float2 x = __ffma2_rn(make_float2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])), c22, nm2);
                return make_float2(ex2_approx(x.x), ex2_approx(x.y));
            };
            float2 zp[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, gp[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            auto sums = [&](const uint32_t (&v)[32]) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float2 e = exp2_of(v, j);
                    zp[j & 1] = __fadd2_rn(zp[j & 1], e);
                    gp[j & 1] = __ffma2_rn(e, make_float2(__uint_as_float(v[16 + 2 * j]), __uint_as_float(v[16 + 2 * j + 1])), gp[j & 1]);
                }
            };
#pragma unroll 1
            for (int q = 0; q < 4; q += 2) {
                tmem_ld_wait32(va);
                tmem_ld16x2_issue(s_tm + 16 * q + 16, s_tm + kTCol + 16 * q + 16, vb);
                sums(va);
                tmem_ld_wait32(vb);
                if (q == 0) tmem_ld16x2_issue(s_tm + 32, s_tm + kTCol + 32, va);
                sums(vb);
            }
            const float lm = tmem_ld1(s_tm + 64);
            tmem_ld16x2_issue(s_tm, s_tm + kTCol, va);
            const float Z = (zp[0].x + zp[0].y) + (zp[1].x + zp[1].y), gt = (gp[0].x + gp[0].y) + (gp[1].x + gp[1].y);
            // the final weight of key j is e_j times one factor per row: alpha / Z in a selected chunk, exp(m - lse) in the
            // local span
            float f, sub = dsum, dl = 0.f;
            if (local) {
                f = __expf(m * s.scale - lse);
            } else {
                const float gc = gt / Z, alpha = __expf(lm * s.scale + bb - lse);
                f = alpha / Z;
                sub = gc;
                dl = alpha * (gc - dsum) * s.scale;
            }
            if (limit < 0) { f = 0.f; sub = 0.f; dl = 0.f; }             // (Z = 0: nothing may leak a NaN)
            const float2 f2 = make_float2(f, f), sc2 = make_float2(s.scale, s.scale), ns2 = make_float2(-sub, -sub);
            auto store = [&](const uint32_t (&v)[32], int q) {           // columns 16 q .. 16 q + 15 of d S and W
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t pd[4], pw[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int i = 4 * h + j;
                        const float2 w = __fmul2_rn(exp2_of(v, i), f2);
                        const float2 t = __fadd2_rn(make_float2(__uint_as_float(v[16 + 2 * i]), __uint_as_float(v[16 + 2 * i + 1])), ns2);
                        const float2 d = __fmul2_rn(__fmul2_rn(w, sc2), t);
                        pd[j] = pack_bf16(d.x, d.y);
                        pw[j] = pack_bf16(w.x, w.y);
                    }
                    const uint32_t at = swz128(row, 2 * q + h);
                    *reinterpret_cast<uint4*>(dsbuf + at) = make_uint4(pd[0], pd[1], pd[2], pd[3]);
                    *reinterpret_cast<uint4*>(wbuf + at) = make_uint4(pw[0], pw[1], pw[2], pw[3]);
                }
            };
            // the previous tile's products have read d S and W
            if (n > 0 && !wait(&sm.done[(n - 1) & 1], ((n - 1) >> 1) & 1)) break;
            dlam_of(grp)[row] = dl;
#pragma unroll 1
            for (int q = 0; q < 4; q += 2) {
                tmem_ld_wait32(va);
                tmem_ld16x2_issue(s_tm + 16 * q + 16, s_tm + kTCol + 16 * q + 16, vb);
                store(va, q);
                tmem_ld_wait32(vb);
                if (q == 0) tmem_ld16x2_issue(s_tm + 32, s_tm + kTCol + 32, va);
                store(vb, q + 1);
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.ds_full[grp]);
        }
    } else if (warp < kGatherWarp) {
        // ================================================================ read-out: d Q rows, d K and d V of a run
        const int rw = warp - kReadWarp;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(rw * 32) << 16);
        uint8_t* stg0 = stgbuf + 2 * rw * kStgBytes;
        const int row = rw * 32 + lane;
        uint32_t run = 0;
        uint2 lmv = make_uint2(0u, 0u);
        for (uint32_t n = 0; tile_of(n); ++n) {
            const Tile& tl = rec[n % kMeta];
            const uint32_t sl = n & 1u;
            const int flags = tl.flags, kv = tl.kv, head0 = tl.head0;
            if (flags & 256) {
                ++run;
                lmv = make_uint2(0u, 0u);
                if (tl.lm >= 0) lmv = __ldg(reinterpret_cast<const uint2*>(a.lm + static_cast<long long>(tl.lm) * kD) + lane);
            }
            // lane x < 8 sends the box of the warp's entry x
            const int e = 8 * rw + (lane & 7), tok = lane < 8 && e < (flags & 255) ? tl.tok0 + (tl.ent[e] >> 8) : -1;
            __syncwarp();
            if (lane == 0) tile_done(n);
            if (!wait(&sm.dq_full, n & 1)) break;
            tc_fence_after_sync();
            // Two copies by turns, each written by all four warps alike: with this tile's d Q complete every warp is through with
            // the tile before the last, so nobody reads the run before the last any more.
            uint8_t* lmt = run & 1u ? reinterpret_cast<uint8_t*>(rec + kMeta) : kbuf + kKBlock + kKHole + kDlamBytes;
            if (flags & 256) *reinterpret_cast<uint2*>(lmt + 8 * lane) = lmv;
            __syncwarp();                            // (also ahead of the loads below, which take the whole warp)
            uint32_t va[32];
            // 32 columns at a time, the borrowed ones first (the first for the even tiles, the last for the odd ones)
            const uint32_t q_tm = t_lane + dq_col(sl);
            const int x0 = sl ? 3 : 0, dx = sl ? -1 : 1;
            tmem_ld32_issue(q_tm + 32 * x0, va);
            const float dl1 = dlam_of(sl)[row];
            const float2 dl = make_float2(dl1, dl1);
#pragma unroll 1
            for (int p = 0; p < 4; ++p) {
                const int x = x0 + dx * p;
                uint4 lp[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) lp[i] = *reinterpret_cast<const uint4*>(lmt + 64 * x + 16 * i);
                tmem_ld_wait32(va);
                if (p == 0 || p == 3) {
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(p == 0 ? &sm.slot_empty[sl] : &sm.dq_empty);
                }
                uint8_t* stg = stg0 + (p & 1) * kStgBytes;
                if (lane < 8) bulk_wait_read<1>();                     // the last piece but one has left its staging rows
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint2 l = i & 1 ? make_uint2(lp[i >> 1].z, lp[i >> 1].w) : make_uint2(lp[i >> 1].x, lp[i >> 1].y);
                    const float2 g0 = __ffma2_rn(dl, make_float2(__uint_as_float(l.x << 16), __uint_as_float(l.x & 0xffff0000u)),
                                                 make_float2(__uint_as_float(va[4 * i]), __uint_as_float(va[4 * i + 1])));
                    const float2 g1 = __ffma2_rn(dl, make_float2(__uint_as_float(l.y << 16), __uint_as_float(l.y & 0xffff0000u)),
                                                 make_float2(__uint_as_float(va[4 * i + 2]), __uint_as_float(va[4 * i + 3])));
                    *reinterpret_cast<float4*>(stg + swz128(lane, i)) = make_float4(g0.x, g0.y, g1.x, g1.y);
                }
                if (p < 3) tmem_ld32_issue(q_tm + 32 * (x + dx), va);
                fence_proxy_async_smem();
                __syncwarp();
                if (tok >= 0) tma_red_add_3d(&map_dq, stg + lane * 512, 32 * x, tok, head0);
                if (lane < 8) bulk_commit();
                __syncwarp();                                            // (the wait for the next piece takes the whole warp)
            }
            if (flags & 512) {
                // ---- the run's last tile: d K^T and d V^T leave tensor memory, a lane per dimension
                if (!wait(&sm.done[sl], (n >> 1) & 1)) break;
                tc_fence_after_sync();
                const long long at = static_cast<long long>(kv) * kD + rw * 32 + lane;
                const int keys = (flags >> 16) & 127;
#pragma unroll 1
                for (int h = 0; h < 4; ++h) {
                    tmem_ld32_issue(t_lane + kDkCol + 32 * h, va);
                    tmem_ld_wait32(va);
                    if (h == 3) {
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sm.acc_empty);
                    }
                    float* dst = (h < 2 ? a.dk : a.dv) + at + static_cast<long long>(h & 1) * 32 * kD;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if ((h & 1) * 32 + j < keys) red_add_f32(dst + j * kD, __uint_as_float(va[j]));
                }
            }
        }
        if (lane < 8) bulk_wait_all();                                   // own copies in flight
    } else if (warp < kLoadWarp) {
        // ================================================================ gather of the Q and dO rows; d landmark
        // (entry-major, head-minor; an instruction copies two 256-byte rows of one entry, see the forward's gather; a warp
        // fills rows 32 gw .. 32 gw + 31 of the tile and sums the same rows for d landmark before it overwrites them)
        const int gw = warp - kGatherWarp, p16 = lane & 15, hh = lane >> 4;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, bacc = 0.f;       // dims 8 p16 .. + 7, rows of half hh
        int fl0 = 0, fl1 = 0;                                                       // flags of the last tile and the one before
        int lr0 = 0, lr1 = 0;                                                       // their landmark rows (-1: none)
        auto landmark_sums = [&](uint32_t n, int fl, int lr) {                                      // tile n: + sum over its rows of (scale d lambda) q
            const uint32_t sl = n & 1u;
            if (!wait(&sm.ds_full[sl], (n >> 1) & 1)) return;
            // (half a warp sums 16 neighbouring rows)
            const float4* dl = reinterpret_cast<const float4*>(dlam_of(sl) + gw * 32 + hh * 16);
            const uint8_t* qt = qbuf + sl * kQBytes + (p16 >> 3) * 16384;
#pragma unroll 1
            for (int r = 0; r < 4; ++r) {
                const float4 d4 = dl[r];
                const float d[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 raw = *reinterpret_cast<const uint4*>(qt + swz128(gw * 32 + hh * 16 + 4 * r + i, p16 & 7));
                    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        acc[2 * x] = fmaf(d[i], __uint_as_float(w[x] << 16), acc[2 * x]);
                        acc[2 * x + 1] = fmaf(d[i], __uint_as_float(w[x] & 0xffff0000u), acc[2 * x + 1]);
                    }
                    bacc += d[i];
                }
            }
            if (fl & 512) {
#pragma unroll
                for (int x = 0; x < 8; ++x) acc[x] += __shfl_xor_sync(kFullMask, acc[x], 16);
                bacc += __shfl_xor_sync(kFullMask, bacc, 16);
                if (lr >= 0) {
                    if (hh == 0) {
                        float* dst = a.dlm + static_cast<long long>(lr) * kD + 8 * p16;
                        red_add_v4(dst, acc[0], acc[1], acc[2], acc[3]);
                        red_add_v4(dst + 4, acc[4], acc[5], acc[6], acc[7]);
                    }
                    if (lane == 0 && a.dbias) red_add_f32(a.dbias + lr, bacc / s.scale);
                }
#pragma unroll
                for (int x = 0; x < 8; ++x) acc[x] = 0.f;
                bacc = 0.f;
            }
        };
        uint32_t end = ~0u;                                              // number of tiles, once known; the sums run two behind
        for (uint32_t n = 0; ok; ++n) {
            if (n < end && !tile_of(n)) end = n;
            if (!ok || (end != ~0u && n >= end + 2)) break;
            const uint32_t sl = n & 1u;
            if (n >= 2) landmark_sums(n - 2, fl1, lr1);
            fl1 = fl0;
            lr1 = lr0;
            if (n >= end) continue;
            const Tile& tl = rec[n % kMeta];
            const int tok = tl.ent[min(8 * gw + (lane & 7), (tl.flags & 255) - 1)] >> 8, row0 = tl.row0;
            fl0 = tl.flags;
            lr0 = tl.lm;
            __syncwarp();
            if (lane == 0) tile_done(n);
            if (n >= 2 && !wait(&sm.done[sl], ((n >> 1) - 1) & 1)) break;
            __syncwarp();
            const uint32_t off = sl * kQBytes + (p16 >> 3) * 16384;
            const uint32_t qa = smem_u32(qbuf) + off, oa = smem_u32(obuf) + off;
            const long long src0 = static_cast<long long>(row0 + hh * hs) * kD + p16 * 8;
#pragma unroll 1
            for (int k0 = 0; k0 < 8; k0 += 4) {
                int tokv[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) tokv[k] = __shfl_sync(kFullMask, tok, k0 + k);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int r = 32 * gw + 4 * k0 + 2 * k;             // rows r, r + 1: heads (r & 3), + 1 of entry r / 4
                    const long long at = src0 + (static_cast<long long>((2 * k) & 3) * hs + tokv[k >> 1]) * kD;
                    const uint32_t d = swz128(r + hh, p16 & 7);
                    cp_async16(qa + d, a.q + at);
                    cp_async16(oa + d, a.dout + at);
                }
            }
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&sm.q_full[sl])) : "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.q_full[sl]);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == kLoadWarp) {
        // ================================================================ K, V and landmark of the runs
        uint32_t run = 0;
        for (uint32_t n = 0; tile_of(n); ++n) {
            const Tile& tl = rec[n % kMeta];
            const int flags = tl.flags, pair = tl.kv / s.T, row = tl.kv - pair * s.T, lmr = tl.lm;
            __syncwarp();
            if (lane == 0) tile_done(n);
            if (!(flags & 256)) continue;
            if (lane == 0) {                                            // (mostly a few tiles ahead: into L2 already)
                tma_prefetch_l2_3d(&map_k, 0, row, pair);
                tma_prefetch_l2_3d(&map_k, 64, row, pair);
                tma_prefetch_l2_3d(&map_v, 0, row, pair);
                tma_prefetch_l2_3d(&map_v, 64, row, pair);
            }
            uint4 lmp = make_uint4(0u, 0u, 0u, 0u);
            if (lane < 16 && lmr >= 0) lmp = *reinterpret_cast<const uint4*>(a.lm + static_cast<long long>(lmr) * kD + lane * 8);
            if (run > 0 && !wait(&sm.k_empty, (run - 1) & 1)) break;
            ++run;
            if (lane == 0) {
                mbar_expect_tx(&sm.k_ready, 16384 + kVBytes);
                tma_load_3d(kbuf, &map_k, &sm.k_ready, 0, row, pair);
                tma_load_3d(kbuf + kKBlock, &map_k, &sm.k_ready, 64, row, pair);
                tma_load_3d(vbuf, &map_v, &sm.k_ready, 0, row, pair);
                tma_load_3d(vbuf + 8192, &map_v, &sm.k_ready, 64, row, pair);
            }
            if (lane < 16) *reinterpret_cast<uint4*>(kbuf + (lane >> 3) * (kKBlock) + swz128(64, lane & 7)) = lmp;
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.k_ready);
        }
        if (run > 0) mbar_wait(&sm.k_ready, (run - 1) & 1);             // own copies in flight
    } else if (warp == kFrontWarp) {
        // ================================================================ S = Q [K; k']^T, T = dO V^T (one thread)
        {
            constexpr uint32_t idesc_s = umma_idesc_bf16(kRows, kNS), idesc_t = umma_idesc_bf16(kRows, kS);
            const uint64_t dk0 = umma_desc_k128(smem_u32(kbuf)), dv0 = umma_desc_k128(smem_u32(vbuf));
            uint32_t run = 0;
            for (uint32_t n = 0; tile_of(n); ++n) {
                const uint32_t sl = __shfl_sync(kFullMask, n & 1u, 0);
                const int flags = rec[n % kMeta].flags;
                __syncwarp();
                if (lane == 0) tile_done(n);
                if (flags & 256) { wait(&sm.k_ready, run & 1); ++run; }
                if (n >= 2) wait(&sm.slot_empty[sl], ((n >> 1) - 1) & 1);
                wait(&sm.q_full[sl], (n >> 1) & 1);
                if (!(ok = __all_sync(kFullMask, ok))) break;           // (one answer per warp: an election follows)
                fence_proxy_async_smem();
                tc_fence_after_sync();
                const uint64_t dq0 = umma_desc_k128(smem_u32(qbuf) + sl * kQBytes), do0 = umma_desc_k128(smem_u32(obuf) + sl * kQBytes);
                const uint32_t d = tmem_base + slot_col(sl);
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        umma_bf16(d, dq0 + (((ks >> 2) * 16384 + (ks & 3) * 32) >> 4), dk0 + (((ks >> 2) * (kKBlock) + (ks & 3) * 32) >> 4),
                                  idesc_s, ks > 0 ? 1u : 0u);
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        umma_bf16(d + kTCol, do0 + (((ks >> 2) * 16384 + (ks & 3) * 32) >> 4), dv0 + (((ks >> 2) * 8192 + (ks & 3) * 32) >> 4),
                                  idesc_t, ks > 0 ? 1u : 0u);
                    umma_commit(&sm.st_full[sl]);
                }
                __syncwarp();
            }
        }
    } else if (warp == kBackWarp) {
        // ================================================================ d Q, d K^T, d V^T (one thread)
        {
            constexpr uint32_t idesc_q = umma_idesc_bf16(kRows, kD) | kUmmaBMnMajor;
            constexpr uint32_t idesc_kv = umma_idesc_bf16(kD, kS) | kUmmaAMnMajor | kUmmaBMnMajor;
            const uint64_t kmn = umma_desc_mn128(smem_u32(kbuf), kKBlock, 1024u);
            const uint64_t dsk = umma_desc_k128(smem_u32(dsbuf));
            const uint64_t dsmn = umma_desc_mn128(smem_u32(dsbuf), 8192u, 1024u), wmn = umma_desc_mn128(smem_u32(wbuf), 8192u, 1024u);
            uint32_t run = 0, n = 0;
            for (; tile_of(n); ++n) {
                const uint32_t sl = __shfl_sync(kFullMask, n & 1u, 0);
                const int flags = rec[n % kMeta].flags;
                const bool first = (flags & 256) != 0;
                __syncwarp();
                if (lane == 0) tile_done(n);
                if (first) { wait(&sm.k_ready, run & 1); ++run; }
                if (n > 0) wait(&sm.dq_empty, (n - 1) & 1);
                wait(&sm.ds_full[sl], (n >> 1) & 1);
                if (!(ok = __all_sync(kFullMask, ok))) break;
                tc_fence_after_sync();
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma_bf16(tmem_base + dq_col(sl), dsk + ((ks * 32) >> 4), kmn + ((ks * 2048) >> 4), idesc_q, ks > 0 ? 1u : 0u);
                    umma_commit(&sm.dq_full);
                    if (flags & 512) umma_commit(&sm.k_empty);
                }
                __syncwarp();
                // the previous run's accumulators have been read
                if (first && run > 1) {
                    wait(&sm.acc_empty, (run - 2) & 1);
                    if (!(ok = __all_sync(kFullMask, ok))) break;
                    tc_fence_after_sync();
                }
                const uint64_t qmn = umma_desc_mn128(smem_u32(qbuf) + sl * kQBytes, 16384u, 1024u);
                const uint64_t omn = umma_desc_mn128(smem_u32(obuf) + sl * kQBytes, 16384u, 1024u);
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint32_t accf = (!first || ks > 0) ? 1u : 0u;
                        umma_bf16(tmem_base + kDkCol, qmn + ((ks * 2048) >> 4), dsmn + ((ks * 2048) >> 4), idesc_kv, accf);
                        umma_bf16(tmem_base + kDvCol, omn + ((ks * 2048) >> 4), wmn + ((ks * 2048) >> 4), idesc_kv, accf);
                    }
                    umma_commit(&sm.done[sl]);
                }
                __syncwarp();
            }
            // every product has completed before tensor memory is freed
            if (n > 0 && ok) wait(&sm.done[(n - 1) & 1], ((n - 1) >> 1) & 1);
        }
    } else {
        // ================================================================ tile records and entries
        // The segments (query blocks, or one pair of each) one after the other, the CTA's share of each; a run is a stretch
        // of the share's tiles on one (pair, chunk).  A lane holds a tile's record; the entries are fetched two tiles ahead.
        uint32_t n = 0;
        int sg = -1;
        long long t = 0, hi = 0;
        int i0 = 0;
        auto put = [&](int flags, int row0, int kv, int lmr, int vis, int head0, int ent) {
            Tile& tl = rec[n % kMeta];
            if (n >= kMeta && !wait(&sm.meta_empty[n % kMeta], ((n / kMeta) - 1) & 1)) return;
            tl.ent[lane] = ent;
            if (lane == 0) { tl.flags = flags; tl.row0 = row0; tl.kv = kv; tl.lm = lmr; tl.vis = vis; tl.head0 = head0; tl.tok0 = i0; }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.meta_full[n % kMeta]);
            ++n;
        };
        while (ok) {
            while (t >= hi && ++sg < a.n_seg) {
                const int t_begin = a.seg_toff[sg], n_tiles = a.seg_toff[sg + 1] - t_begin;
                i0 = sg / a.segs * a.qb;
                t = t_begin + static_cast<long long>(blockIdx.x) * n_tiles / gridDim.x;
                hi = t_begin + static_cast<long long>(blockIdx.x + 1) * n_tiles / gridDim.x;
            }
            if (t >= hi) break;
            int4 prev = make_int4(-1, -1, 0, 0);
            for (; t < hi && ok; t += 32) {
                // lane x: record and flags of tile t + x
                const int nb = static_cast<int>(hi - t < 32 ? hi - t : 32);
                const int4 rec = lane < nb ? a.tiles[t + lane] : make_int4(-1, -1, 0, 0);
                const int4 after = t + 32 < hi ? a.tiles[t + 32] : make_int4(-1, -1, 0, 0);
                int px = __shfl_up_sync(kFullMask, rec.x, 1), py = __shfl_up_sync(kFullMask, rec.y, 1);
                int nx = __shfl_down_sync(kFullMask, rec.x, 1), ny = __shfl_down_sync(kFullMask, rec.y, 1);
                if (lane == 0) { px = prev.x; py = prev.y; }
                if (lane == 31) { nx = after.x; ny = after.y; }
                const int b = rec.x / s.Hkv, gk = rec.x - b * s.Hkv, c = rec.y;
                const int head0 = b * s.Hq + gk * kG, row0 = head0 * hs + i0, kv = rec.x * s.T + c * kS;
                const int lmr = c < s.C ? (b * s.Hl + gk) * s.C + c : -1, vis = s.pos0 + i0 - c * kS;     // (B Hkv C < 2^24)
                const int flags = min(kS, s.T - c * kS) << 16 | rec.w | (rec.x != px || rec.y != py ? 256 : 0) | (rec.x != nx || rec.y != ny ? 512 : 0);
                int e0 = a.entries[t * kTok + lane], e1 = nb > 1 ? a.entries[(t + 1) * kTok + lane] : 0;
#pragma unroll 1
                for (int x = 0; x < nb && ok; ++x) {
                    const int e2 = x + 2 < nb ? a.entries[(t + x + 2) * kTok + lane] : 0;
                    put(__shfl_sync(kFullMask, flags, x), __shfl_sync(kFullMask, row0, x), __shfl_sync(kFullMask, kv, x),
                        __shfl_sync(kFullMask, lmr, x), __shfl_sync(kFullMask, vis, x), __shfl_sync(kFullMask, head0, x), e0);
                    e0 = e1;
                    e1 = e2;
                }
                prev.x = __shfl_sync(kFullMask, rec.x, 31);
                prev.y = __shfl_sync(kFullMask, rec.y, 31);
            }
            t = hi;
        }
#pragma unroll 1
        for (int x = 0; x < 2; ++x)                                     // (one for either statistics group)
            if (ok) put(0, 0, 0, 0, 0, 0, 0);
    }
    if (!ok && lane == 0) set_status(a.status, kDevTimeout);
    __syncwarp();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == kFrontWarp) tmem_dealloc(tmem_base, 512);
}

// D = dout . out per row: half a warp per row.
__global__ void __launch_bounds__(256) backward_dsum_kernel(const uint4* dout, const uint4* out, float* dsum, long long rows) {
    const int lane = threadIdx.x & 15;
    const long long step = static_cast<long long>(gridDim.x) * 16;
    for (long long row = static_cast<long long>(blockIdx.x) * 16 + (threadIdx.x >> 4); row < rows + (rows & 1); row += step) {
        const long long r = row < rows ? row : rows - 1;               // (both halves of a warp take part in the sums)
        const uint4 x = __ldcs(dout + r * 16 + lane), y = __ldcs(out + r * 16 + lane);
        const uint32_t xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
        float acc = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc = fmaf(__uint_as_float(xv[i] << 16), __uint_as_float(yv[i] << 16), acc);
            acc = fmaf(__uint_as_float(xv[i] & 0xffff0000u), __uint_as_float(yv[i] & 0xffff0000u), acc);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(kFullMask, acc, o);
        if (lane == 0 && row < rows) dsum[row] = acc;
    }
}

size_t dsum_bytes(const Shape& s) { return (static_cast<size_t>(s.B) * s.Hq * s.R * sizeof(float) + 255) / 256 * 256; }

}  // namespace

// The swizzled tiles start on multiples of 1024 bytes if the kernel's dynamic shared memory does, which lies behind what the system
// reserves (1024 bytes) and the kernel's static part (none).  Where a toolchain lays this out in another way the generic kernel
// takes the calls.  (Asked once per device; true where no device answers, e.g. a workspace-size query on a host without a GPU.)
static bool tiles_aligned() {
    static int known[64] = {};                   // 1: aligned, 2: not
    const int dev = PerDeviceOnce::device();
    if (dev < 0) return true;
    if (known[dev] == 0) {
        int reserved = 0;
        cudaFuncAttributes attr;
        if (cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
            cudaFuncGetAttributes(&attr, backward_tc_kernel) != cudaSuccess)
            return true;
        known[dev] = (static_cast<size_t>(reserved) + attr.sharedSizeBytes) % 1024 == 0 ? 1 : 2;
    }
    return known[dev] == 1;
}

bool prefill_backward_fast_supports(const Shape& s, int dtype) {
    return prefill_fast_supports(s, dtype) && tiles_aligned() && s.Hl == s.Hkv && s.K + 17 <= 255 &&
           static_cast<long long>(s.B) * s.Hq * s.R < (1ll << 31);
}

size_t prefill_backward_fast_scratch_bytes(const Shape& s) { return dsum_bytes(s) + inverse_index_bytes(s); }

int launch_prefill_backward_fast(const Shape& s, const BackwardTensors& t, cudaStream_t stream) {
    if (t.scratch_bytes < prefill_backward_fast_scratch_bytes(s)) return HILS_ERR_WORKSPACE;
    char* sc = static_cast<char*>(t.scratch);
    float* dsum = reinterpret_cast<float*>(sc);
    const long long rows = static_cast<long long>(s.B) * s.Hq * s.R;
    const long long want = (rows + 15) / 16;
    const unsigned blocks = static_cast<unsigned>(want < 16ll * sm_count() ? want : 16ll * sm_count());
    backward_dsum_kernel<<<blocks, 256, 0, stream>>>(static_cast<const uint4*>(t.dout), static_cast<const uint4*>(t.out), dsum, rows);
    if (cudaGetLastError() != cudaSuccess) return HILS_ERR_CUDA;
    trace_mark("backward_dsum", stream);
    InverseIndex ix;
    const int rc = build_inverse_index(s, t.sel_idx, sc + dsum_bytes(s), t.scratch_bytes - dsum_bytes(s), &ix, stream);
    if (rc < 0) return rc;
    CUtensorMap map_k, map_v, map_dq;
    const uint64_t kv_pairs = static_cast<uint64_t>(s.B) * s.Hkv;
    if (!make_kv_map(&map_k, t.k, kv_pairs, s.T, s.pos0 + s.R, kD, 64, kS) || !make_kv_map(&map_v, t.v, kv_pairs, s.T, s.pos0 + s.R, kD, 64, kS) ||
        !make_f32_rows_map(&map_dq, t.dq, static_cast<uint64_t>(s.B) * s.Hq, s.R, kD, 32, kG))
        return HILS_ERR_CUDA;
    static PerDeviceOnce attr_once;
    if (attr_once.pending()) {
        if (cudaFuncSetAttribute(backward_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemBytes)) != cudaSuccess)
            return HILS_ERR_CUDA;
        attr_once.done();
    }
    // One (query block, pair) at a time where that gives every CTA some 24 tiles (each segment ends with a drained pipeline
    // and two cut runs), else all pairs of a block together.
    const int pairs = s.B * s.Hkv, toks = s.R < ix.qb ? s.R : ix.qb;
    const bool by_pair = static_cast<long long>(toks) * (s.K + 1) >= 24ll * ix.tile_tok * sm_count();
    BArgs a;
    a.s = s;
    a.q = static_cast<const __nv_bfloat16*>(t.q);
    a.dout = static_cast<const __nv_bfloat16*>(t.dout);
    a.lm = static_cast<const __nv_bfloat16*>(t.landmarks);
    a.bias = t.bias;
    a.lse = t.lse;
    a.dsum = dsum;
    a.entries = ix.entries;
    a.tiles = ix.tiles;
    a.seg_toff = by_pair ? ix.pair_toff : ix.blk_toff;
    a.segs = by_pair ? pairs : 1;
    a.n_seg = ix.n_blocks * a.segs;
    a.qb = ix.qb;
    a.dq = t.dq;
    a.dk = t.dk;
    a.dv = t.dv;
    a.dlm = t.dlandmarks;
    a.dbias = t.dbias;
    a.status = t.status;
    if (launch_pdl(backward_tc_kernel, dim3(sm_count()), dim3(kThreads), kSmemBytes, stream, map_k, map_v, map_dq, a) != cudaSuccess)
        return HILS_ERR_CUDA;
    trace_mark("backward_attend", stream);
    return rc + 2;
}

}  // namespace hils
