// Chunk summaries (Proposition 3.1, Eq. prop_q_c): k'_c = Attn(q'_c, K_c, K_c) and b'_c = entropy of the
// attention distribution of the chunk's learnable query over the chunk's keys.
//
// One warp per (sequence, landmark head, chunk).  The warp copies the chunk's keys into its own padded
// shared-memory tile with cp.async (every key byte is read from memory exactly once, 16 bytes per lane,
// coalesced), then
//   scores      lane l owns key rows l, l + 32, ...: a full dot product per row from shared memory (rows are
//               272-byte apart for d = 128 bf16, so a quarter warp touches all 32 banks once), no shuffles;
//   softmax     two warp reductions; b' = log Z - sum p (s - max);
//   k'          lane l owns d/32 output dimensions and runs over the rows.
// The loops are rolled (a first, fully unrolled register version reached 20 % of the memory bandwidth).  The kernel is bound by HBM: algorithmic bytes = the keys of the summarised chunks.
#include "internal.h"
#include "tma.cuh"

namespace hils {
namespace {

constexpr int kMaxS = 128;
constexpr int kMaxWarps = 4;

struct LArgs {
    int B, Hkv, Hl, C, S;
    long long T;
    float scale;
    const void* lq;
    const void* k;
    const int32_t* seq;
    void* lm;
    float* bias;
    int c0, cn;
};

__device__ __forceinline__ float elem_f32(float x) { return x; }
__device__ __forceinline__ float elem_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void elem_set(float& dst, float x) { dst = x; }
__device__ __forceinline__ void elem_set(__nv_bfloat16& dst, float x) { dst = __float2bfloat16_rn(x); }

// D = head dimension (32, 64, 128, 256).  Shared memory per warp: S rows of D * sizeof(T) + 16 bytes, D floats
// for the scaled query and kMaxS floats for the probabilities.
template <typename T, int D>
__global__ void landmark_summary_kernel(const LArgs a) {
    extern __shared__ __align__(16) uint8_t lsm[];
    constexpr int RB = D * static_cast<int>(sizeof(T));       // bytes per key row
    constexpr int RS = RB + 16;                               // row stride in shared memory
    constexpr int EPP = 16 / static_cast<int>(sizeof(T));     // elements per 16-byte piece
    constexpr int VPL = D / 32;                               // output dimensions per lane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const size_t per_warp = static_cast<size_t>(a.S) * RS + D * sizeof(float) + kMaxS * sizeof(float);
    uint8_t* tile = lsm + warp * per_warp;
    float* qs = reinterpret_cast<float*>(tile + static_cast<size_t>(a.S) * RS);
    float* ps = qs + D;
    const long long item = static_cast<long long>(blockIdx.x) * nwarps + warp;
    const long long total = static_cast<long long>(a.B) * a.Hl * a.cn;
    if (item >= total) return;
    const int c = a.c0 + static_cast<int>(item % a.cn);
    const int hl = static_cast<int>((item / a.cn) % a.Hl);
    const int b = static_cast<int>(item / (static_cast<long long>(a.cn) * a.Hl));
    const int hkv = hl / (a.Hl / a.Hkv);
    long long len = a.seq ? a.seq[b] : a.T;
    len = len < 0 ? 0 : (len > a.T ? a.T : len);
    const long long j0 = static_cast<long long>(c) * a.S;
    const int n = static_cast<int>(len - j0 < 0 ? 0 : (len - j0 > a.S ? a.S : len - j0));
    const long long orow = (static_cast<long long>(b) * a.Hl + hl) * a.C + c;
    T* out = static_cast<T*>(a.lm) + orow * D + lane * VPL;
    if (n == 0) {
#pragma unroll
        for (int i = 0; i < VPL; ++i) elem_set(out[i], 0.f);
        if (lane == 0) a.bias[orow] = 0.f;
        return;
    }
    // ---- the chunk's keys -> shared memory (asynchronously), the scaled query meanwhile
    {
        const uint8_t* src = reinterpret_cast<const uint8_t*>(
            static_cast<const T*>(a.k) + ((static_cast<long long>(b) * a.Hkv + hkv) * a.T + j0) * D);
        constexpr int PPR = RB / 16;
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(tile));
        for (int x = lane; x < n * PPR; x += 32) {
            const int row = x / PPR, pc = x % PPR;
            cp_async16(dst + row * RS + pc * 16, src + static_cast<size_t>(row) * RB + pc * 16);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        const T* q = static_cast<const T*>(a.lq) + orow * D;
        for (int e = lane; e < D; e += 32) qs[e] = elem_f32(q[e]) * a.scale;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    // ---- scores s_j = scale * q'_c . k_j for the rows of this lane (slot r: row lane + 32 r)
    float sreg[kMaxS / 32];
#pragma unroll
    for (int r = 0; r < kMaxS / 32; ++r) {
        sreg[r] = -INFINITY;
        const int j = lane + 32 * r;
        if (j < n) {
            const uint8_t* row = tile + static_cast<size_t>(j) * RS;
            float s = 0.f;
#pragma unroll 4
            for (int pc = 0; pc < RB / 16; ++pc) {
                const uint4 raw = *reinterpret_cast<const uint4*>(row + pc * 16);
                const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
                for (int i = 0; i < EPP; ++i) s = fmaf(qs[pc * EPP + i], elem_f32(e[i]), s);
            }
            sreg[r] = s;
        }
    }
    // ---- p = softmax(s), b' = -sum p log p = log Z - sum p (s - m)
    float m = -INFINITY;
#pragma unroll
    for (int r = 0; r < kMaxS / 32; ++r) m = fmaxf(m, sreg[r]);
    m = warp_max(m);
    float z = 0.f, pe[kMaxS / 32];
#pragma unroll
    for (int r = 0; r < kMaxS / 32; ++r) {
        pe[r] = sreg[r] == -INFINITY ? 0.f : __expf(sreg[r] - m);
        z += pe[r];
    }
    z = warp_sum(z);
    const float zi = 1.f / z;
    float psum = 0.f;
#pragma unroll
    for (int r = 0; r < kMaxS / 32; ++r) {
        const float pj = pe[r] * zi;
        if (pj > 0.f) psum = fmaf(pj, sreg[r] - m, psum);
        if (lane + 32 * r < n) ps[lane + 32 * r] = pj;
    }
    psum = warp_sum(psum);
    __syncwarp();
    // ---- k' = sum_j p_j k_j: this lane's VPL output dimensions over all rows
    float acc[VPL];
#pragma unroll
    for (int i = 0; i < VPL; ++i) acc[i] = 0.f;
    const uint8_t* col = tile + lane * VPL * sizeof(T);
#pragma unroll 8
    for (int j = 0; j < n; ++j) {
        const float pj = ps[j];
        const T* e = reinterpret_cast<const T*>(col + static_cast<size_t>(j) * RS);
#pragma unroll
        for (int i = 0; i < VPL; ++i) acc[i] = fmaf(pj, elem_f32(e[i]), acc[i]);
    }
#pragma unroll
    for (int i = 0; i < VPL; ++i) elem_set(out[i], acc[i]);
    if (lane == 0) a.bias[orow] = __logf(z) - psum;
}

// ---- bf16, d = 128, S = 64, at most 8 landmark heads per KV head: both contractions on mma.sync ----
// Persistent: one CTA of 14 warps per SM.  A warp owns a 16 KB stage and takes every 14th (sequence, KV head, chunk) item of
// the CTA: the keys arrive by TMA, and the next item's are requested as soon as this one's have been read.
// S^T = K q'^T with the keys in the MMA rows and the landmark heads of the KV head in its columns, then k'^T = K^T P^T
// with P split into two bf16 terms (p = hi + lo), so that the weights keep 16 bits of mantissa.
// Bound: HBM, reached by the number of warps (an item takes a warp 2 us of dependent steps): 8 x 64K ragged tokens, 8 KV
// heads: 168 us with a CTA per four chunks (load, compute, leave), 155 with 7 warps of two stages, 122 (6.1 TB/s) with 14.
constexpr int kTcWarps = 14;
constexpr int kTcTileBytes = 64 * 128 * 2;


__global__ void __launch_bounds__(kTcWarps * 32, 1)
landmark_summary_tc_kernel(const __grid_constant__ CUtensorMap map_k, const LArgs a) {
    extern __shared__ uint8_t lsm_raw[];
    __shared__ uint64_t full[kTcWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    uint8_t* tile = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(lsm_raw) + 1023) & ~uintptr_t(1023)) + warp * kTcTileBytes;
    const uint32_t addr = smem_u32(tile);
    uint64_t* bar = &full[warp];
    const int per = a.Hl / a.Hkv;                              // landmark heads per KV head (MMA columns), <= 8
    const int total = a.B * a.Hkv * a.cn;
    __nv_bfloat16* lm = static_cast<__nv_bfloat16*>(a.lm);
    struct Item { int b, hkv, c, n; };
    auto item_of = [&](int k) {                                // item k of this CTA
        Item it;
        const int x = blockIdx.x + k * static_cast<int>(gridDim.x), u = x / a.cn;
        it.c = a.c0 + (x - u * a.cn);
        it.b = u / a.Hkv;
        it.hkv = u - it.b * a.Hkv;
        long long len = a.seq ? a.seq[it.b] : a.T;
        len = len < 0 ? 0 : (len > a.T ? a.T : len);
        const long long left = len - static_cast<long long>(it.c) * 64;
        it.n = static_cast<int>(left < 0 ? 0 : (left > 64 ? 64 : left));
        return it;
    };
    auto out_row = [&](const Item& it) { return (static_cast<long long>(it.b) * a.Hl + it.hkv * per) * a.C + it.c; };    // head 0
    auto request = [&](const Item& it) {                       // one lane
        if (it.n == 0) return;
        const int row = static_cast<int>((static_cast<long long>(it.b) * a.Hkv + it.hkv) * a.T + static_cast<long long>(it.c) * 64);
        mbar_expect_tx(bar, kTcTileBytes);
        tma_load_2d(tile, &map_k, bar, 0, row);
        tma_load_2d(tile + 8192, &map_k, bar, 64, row);
    };
    const int n_items = (total - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
    if (lane == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
    }
    pdl_wait();
    pdl_launch_dependents();
    if (warp >= n_items) return;
    Item cur = item_of(warp);
    if (lane == 0) request(cur);
    __syncwarp();
    uint32_t phase = 0u;
    for (int k = warp; k < n_items; k += kTcWarps) {
        const Item next = k + kTcWarps < n_items ? item_of(k + kTcWarps) : Item{0, 0, 0, 0};
        const long long orow0 = out_row(cur);
        uint32_t q[8][2];                                      // column g: landmark head g of the KV head
        {
            const bool ok = cur.n > 0 && g < per;
            const __nv_bfloat16* row = static_cast<const __nv_bfloat16*>(a.lq) + (orow0 + static_cast<long long>(ok ? g : 0) * a.C) * 128;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                q[ks][0] = ok ? *reinterpret_cast<const uint32_t*>(row + ks * 16 + 2 * t) : 0u;
                q[ks][1] = ok ? *reinterpret_cast<const uint32_t*>(row + ks * 16 + 8 + 2 * t) : 0u;
            }
        }
        if (cur.n == 0) {
            for (int y = lane; y < per * 64; y += 32)
                *reinterpret_cast<uint32_t*>(lm + (orow0 + static_cast<long long>(y >> 6) * a.C) * 128 + (y & 63) * 2) = 0u;
            if (lane < per) a.bias[orow0 + static_cast<long long>(lane) * a.C] = 0.f;
        }
        float o[8][4], bias[2] = {0.f, 0.f};
        if (cur.n > 0) {
            if (!mbar_wait(bar, phase)) {
                // the bounded wait ran out (never seen: the copy has a valid map): mark the chunk's bias NaN and leave
                if (lane < per) a.bias[orow0 + static_cast<long long>(lane) * a.C] = __int_as_float(0x7fc00000);
                return;
            }
            phase ^= 1u;
            const int n = cur.n;
            if (n < 64) {
                // rows past the sequence end may hold anything: zero them before they meet probabilities of 0
                for (int y = lane; y < (64 - n) * 16; y += 32) {
                    const int row = n + (y >> 4), piece = y & 15;
                    *reinterpret_cast<uint4*>(tile + (piece >> 3) * 8192 + swz128(row, piece & 7)) = make_uint4(0u, 0u, 0u, 0u);
                }
                __syncwarp();
                fence_proxy_async_smem();                      // (the stage is overwritten by a bulk copy later)
            }
            float sc[4][4];
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) sc[mt][0] = sc[mt][1] = sc[mt][2] = sc[mt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) {
                    const int row = mt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8, dim = ks * 16 + (lane >> 4) * 8;
                    uint32_t fr[4];
                    ldmatrix_x4(addr + (dim >> 6) * 8192 + swz128(row, (dim & 63) >> 3), fr[0], fr[1], fr[2], fr[3]);
                    mma_bf16_16816(sc[mt], fr, q[ks][0], q[ks][1]);
                }
            // columns 2 t, 2 t + 1; rows (keys) 16 mt + g, + 8
            uint32_t hi[4][2], lo[4][2];
            float p[4][4];
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                float m = -INFINITY;
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) {
                    sc[mt][y] = mt * 16 + g < n ? sc[mt][y] * a.scale : -INFINITY;
                    sc[mt][2 + y] = mt * 16 + 8 + g < n ? sc[mt][2 + y] * a.scale : -INFINITY;
                    m = fmaxf(m, fmaxf(sc[mt][y], sc[mt][2 + y]));
                }
#pragma unroll
                for (int x = 4; x < 32; x <<= 1) m = fmaxf(m, __shfl_xor_sync(kFullMask, m, x));
                float z = 0.f, ps = 0.f;                       // ps = sum e (s - m)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float& s_ = sc[i >> 1][(i & 1) * 2 + y];
                    const float e = __expf(s_ - m);
                    z += e;
                    if (e > 0.f) ps = fmaf(e, s_ - m, ps);
                    p[i >> 1][(i & 1) * 2 + y] = e;
                }
#pragma unroll
                for (int x = 4; x < 32; x <<= 1) {
                    z += __shfl_xor_sync(kFullMask, z, x);
                    ps += __shfl_xor_sync(kFullMask, ps, x);
                }
                const float zi = 1.f / z;
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) { p[mt][y] *= zi; p[mt][2 + y] *= zi; }
                bias[y] = __logf(z) - ps * zi;
            }
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const __nv_bfloat16 h0 = __float2bfloat16_rn(p[mt][2 * h]), h1 = __float2bfloat16_rn(p[mt][2 * h + 1]);
                    const float f0 = __bfloat162float(h0), f1 = __bfloat162float(h1);
                    hi[mt][h] = movmatrix_trans(pack_bf16(f0, f1));
                    lo[mt][h] = movmatrix_trans(pack_bf16(p[mt][2 * h] - f0, p[mt][2 * h + 1] - f1));
                }
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int mt = 0; mt < 8; ++mt) {
                    const int row = kk * 16 + (lane >> 4) * 8 + (lane & 7), dim = mt * 16 + ((lane >> 3) & 1) * 8;
                    uint32_t fr[4];
                    ldmatrix_x4_trans(addr + (dim >> 6) * 8192 + swz128(row, (dim & 63) >> 3), fr[0], fr[1], fr[2], fr[3]);
                    mma_bf16_16816(o[mt], fr, hi[kk][0], hi[kk][1]);
                    mma_bf16_16816(o[mt], fr, lo[kk][0], lo[kk][1]);
                }
        }
        __syncwarp();                                          // every lane has read the stage
        if (lane == 0) request(next);
        if (cur.n > 0) {
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const int h = 2 * t + y;
                if (h < per) {
                    const long long row = orow0 + static_cast<long long>(h) * a.C;
#pragma unroll
                    for (int mt = 0; mt < 8; ++mt) {
                        lm[row * 128 + mt * 16 + g] = __float2bfloat16_rn(o[mt][y]);
                        lm[row * 128 + mt * 16 + 8 + g] = __float2bfloat16_rn(o[mt][2 + y]);
                    }
                    if (g == 0) a.bias[row] = bias[y];
                }
            }
        }
        cur = next;
    }
}

template <typename T, int D>
int launch_one(const LArgs& a, cudaStream_t stream) {
    const long long total = static_cast<long long>(a.B) * a.Hl * a.cn;
    if (total == 0) return 0;
    const size_t per_warp = static_cast<size_t>(a.S) * (D * sizeof(T) + 16) + D * sizeof(float) + kMaxS * sizeof(float);
    int nw = static_cast<int>(69632 / per_warp);            // three 68 KB blocks per SM
    nw = nw < 1 ? 1 : (nw > kMaxWarps ? kMaxWarps : nw);
    const size_t smem = per_warp * nw;
    if (smem > 227 * 1024) return HILS_ERR_UNSUPPORTED;
    static size_t attr_bytes = 0;                             // per instantiation
    if (smem > attr_bytes) {
        if (cudaFuncSetAttribute(landmark_summary_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(smem)) != cudaSuccess)
            return HILS_ERR_CUDA;
        attr_bytes = smem;
    }
    const long long blocks = (total + nw - 1) / nw;
    if (blocks > 0x7fffffffll) return HILS_ERR_UNSUPPORTED;
    landmark_summary_kernel<T, D><<<static_cast<unsigned>(blocks), nw * 32, smem, stream>>>(a);
    return cudaGetLastError() == cudaSuccess ? 1 : HILS_ERR_CUDA;
}

template <typename T>
int launch_typed(const LArgs& a, int d, cudaStream_t stream) {
    switch (d) {
        case 32: return launch_one<T, 32>(a, stream);
        case 64: return launch_one<T, 64>(a, stream);
        case 128: return launch_one<T, 128>(a, stream);
        case 256: return launch_one<T, 256>(a, stream);
        default: return HILS_ERR_UNSUPPORTED;
    }
}

}  // namespace

bool landmark_summary_supports(int d, int S) { return (d == 32 || d == 64 || d == 128 || d == 256) && S >= 1 && S <= kMaxS; }

int launch_landmark_summary(int dtype, int B, int Hkv, int Hl, int C, int d, int S, long long T, float scale,
                            const void* lq, const void* k, const int32_t* seq_lens, int c0, int cn, void* landmarks,
                            float* bias, cudaStream_t stream) {
    LArgs a{B, Hkv, Hl, C, S, T, scale, lq, k, seq_lens, landmarks, bias, c0, cn};
    static const bool no_tc = [] { const char* e = getenv("HILS_LANDMARK_NO_MMA"); return e && e[0] == '1'; }();
    const long long rows = static_cast<long long>(B) * Hkv * T;
    if (!no_tc && dtype == HILS_BF16 && d == 128 && S == 64 && Hl / Hkv <= 8 && rows < (1ll << 31) &&
        static_cast<long long>(B) * Hkv * cn < (1ll << 31)) {
        const long long total = static_cast<long long>(B) * Hkv * cn;
        if (total == 0) return 0;
        CUtensorMap map_k;
        if (!make_bf16_2d_map(&map_k, k, static_cast<uint64_t>(rows), 128, 64, 64)) return HILS_ERR_CUDA;
        const size_t smem = kTcWarps * kTcTileBytes + 1024;
        static PerDeviceOnce attr_once;
        if (attr_once.pending()) {
            if (cudaFuncSetAttribute(landmark_summary_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(smem)) != cudaSuccess)
                return HILS_ERR_CUDA;
            attr_once.done();
        }
        const unsigned blocks = static_cast<unsigned>(total < sm_count() ? total : sm_count());
        // (launched so that a call's start overlaps the end of the kernel before it: calls of 4 x 1.7K tokens back to back 7.8 -> 7.2 us; 8 x 64K
        // tokens take 125 either way, to 0.6 %)
        return launch_pdl(landmark_summary_tc_kernel, dim3(blocks), dim3(kTcWarps * 32), smem, stream, map_k, a) == cudaSuccess ? 1 : HILS_ERR_CUDA;
    }
    return dtype == HILS_F32 ? launch_typed<float>(a, d, stream) : launch_typed<__nv_bfloat16>(a, d, stream);
}

}  // namespace hils
