// Shape-agnostic HiLS kernels on CUDA cores: one warp per (sequence, KV group, query row) for scoring + top-K
// selection, one CTA per (sequence, query head, query row) for attention, its warps sharing the row's chunks.
// They cover fp32 and bf16, any head dim that is a multiple of 32 (<= 256), any chunk size and any local window,
// prefill and decode.  They are the correctness anchor and the fall-back for shapes the tensor-core /
// bandwidth-tuned kernels do not take.
// Bound: the load path.  Every row reads its own K and V rows through L1, so a warp request has to cover whole
// 64-byte runs: four lanes share a key (16-byte pieces, the quad's sum by two shuffles, the query in registers), where a
// lane per key touched 32 lines per request; and a warp takes one chunk, where one warp walked all of a row's chunks.
// fp32, 2048 tokens, d = 64, K = 4: 82 -> 38 us (attention by rows), 16 -> 10 us (selection).
#include "internal.h"
#include "tma.cuh"

namespace hils {
namespace {

constexpr int kWarpsPerBlock = 4;

struct GArgs {
    Shape s;
    const void* q;
    const void* q_route;   // routing query for the surrogate scores (= q unless a separate one was given)
    const void* k;
    const void* v;
    const void* lm;
    const float* bias;
    const int32_t* seq_lens;
    void* out;
    float* lse;
    int32_t* sel;
    int* status;
};

// Position of query row r of sequence b, or -1 if the decode length is invalid.
// The kernels are short, and a division is some forty instructions that are fetched cold: chunks of 64 tokens go by a shift, indexes are
// 32 bits wide (launch_dim holds the rows below 2^31).  2048 tokens, one head, d = 64, K = 4: 30.7 -> 29.4 us.
__host__ __device__ inline int div_chunk(const Shape& s, int x) { return s.S == 64 ? x >> 6 : x / s.S; }                // x >= 0
__device__ inline int left_chunks(const Shape& s, int pos) { return pos < s.W ? 0 : div_chunk(s, pos - s.W + 1); }       // chunks left of the window

__device__ inline int row_position(const GArgs& a, int b, int r) {
    if (!a.s.is_decode) return a.s.pos0 + r;
    const int n = a.seq_lens[b];
    if (n < 1 || n > a.s.T) return -1;
    return n - 1;
}

// One 16-byte piece of a row, widened.
template <typename T> struct Piece;
template <> struct Piece<float> {
    static constexpr int kElems = 4;
    __device__ static void load(const float* p, float (&x)[4]) {
        const float4 a = *reinterpret_cast<const float4*>(p);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
    }
};
template <> struct Piece<__nv_bfloat16> {
    static constexpr int kElems = 8;
    __device__ static void load(const __nv_bfloat16* p, float (&x)[8]) { load8(p, x); }
};

// A quad of lanes shares a row of D elements at most: lane j of the quad owns the 16-byte pieces j, j + 4, ..., npl of
// them.  X: the head dimension is D itself (offsets inside a row are constants).
template <typename T, int D, bool X>
struct Quad {
    static constexpr int kE = Piece<T>::kElems, kPl = D / kE / 4;
    float x[kPl][kE];

    __device__ __forceinline__ static int dim(int d) { return X ? D : d; }
    // row: this lane's first piece
    __device__ __forceinline__ void load(const T* row, int d) {
#pragma unroll
        for (int i = 0; i < kPl; ++i) {
            if (X || i < d / (4 * kE)) {
                Piece<T>::load(row + 4 * kE * i, x[i]);
            } else {
#pragma unroll
                for (int e = 0; e < kE; ++e) x[i][e] = 0.f;
            }
        }
    }
    __device__ __forceinline__ void fill(float v) {
#pragma unroll
        for (int i = 0; i < kPl; ++i)
#pragma unroll
            for (int e = 0; e < kE; ++e) x[i][e] = v;
    }
    // dot product over the quad (the sum in all four lanes)
    __device__ __forceinline__ float dot(const Quad& o) const {
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int i = 0; i < kPl; ++i)
#pragma unroll
            for (int e = 0; e < kE; e += 2) {
                a0 = fmaf(x[i][e], o.x[i][e], a0);
                a1 = fmaf(x[i][e + 1], o.x[i][e + 1], a1);
            }
        a0 += a1;
        a0 += __shfl_xor_sync(kFullMask, a0, 1);
        a0 += __shfl_xor_sync(kFullMask, a0, 2);
        return a0;
    }
    __device__ __forceinline__ void scale_by(float f) {
#pragma unroll
        for (int i = 0; i < kPl; ++i)
#pragma unroll
            for (int e = 0; e < kE; ++e) x[i][e] *= f;
    }
    __device__ __forceinline__ void add_scaled(float f, const Quad& o) {
#pragma unroll
        for (int i = 0; i < kPl; ++i)
#pragma unroll
            for (int e = 0; e < kE; ++e) x[i][e] = fmaf(f, o.x[i][e], x[i][e]);
    }
};

// Insert key x into the descending list held as lst[j] of lane l <-> index j*32+l, keeping K entries.
template <int NR>
__device__ inline void list_insert(unsigned long long (&lst)[NR], unsigned long long x, int K, int lane) {
    int pos = 0;
#pragma unroll
    for (int j = 0; j < NR; ++j) pos += __popc(__ballot_sync(kFullMask, lst[j] > x));
#pragma unroll
    for (int j = NR - 1; j >= 0; --j) {
        const int idx = j * 32 + lane;
        unsigned long long up = __shfl_up_sync(kFullMask, lst[j], 1);
        unsigned long long carry = 0ull;
        if (j > 0) carry = __shfl_sync(kFullMask, lst[j - 1], 31);
        if (lane == 0) up = carry;
        unsigned long long nv = idx < pos ? lst[j] : (idx == pos ? x : up);
        if (idx >= K) nv = 0ull;
        lst[j] = nv;
    }
}
// Merges 32 keys (one per lane, any order) into the list: sorted across the warp, the larger of each list entry and
// its mirror image taken, the bitonic result merged.
template <int NR>
__device__ inline void list_merge(unsigned long long (&lst)[NR], unsigned long long x, int K, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const unsigned long long o = __shfl_xor_sync(kFullMask, x, j);
            const bool upper = (lane & j) != 0, desc = (lane & k) == 0;
            x = (upper != desc) == (x > o) ? x : o;
        }
    const unsigned long long rev = __shfl_xor_sync(kFullMask, x, 31);
    lst[NR - 1] = lst[NR - 1] > rev ? lst[NR - 1] : rev;
#pragma unroll
    for (int h = NR >> 1; h > 0; h >>= 1)
#pragma unroll
        for (int i = 0; i < NR; ++i)
            if ((i & h) == 0) {
                const unsigned long long a = lst[i], b = lst[i + h];
                lst[i] = a > b ? a : b;
                lst[i + h] = a > b ? b : a;
            }
#pragma unroll
    for (int j = 16; j > 0; j >>= 1)
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const unsigned long long o = __shfl_xor_sync(kFullMask, lst[i], j);
            const bool upper = (lane & j) != 0;
            lst[i] = upper == (lst[i] < o) ? lst[i] : o;
        }
#pragma unroll
    for (int i = 0; i < NR; ++i)
        if (i * 32 + lane >= K) lst[i] = 0ull;
}

// Scoring (Eq. surrogate top-k, per head), group max (App. C) and exact top-K with ties to the
// lower chunk id.  One warp per (b, g, r), 32 chunks at a time.
template <typename T, int D, bool X, int NR>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
generic_select_kernel(const GArgs a) {
    const Shape& s = a.s;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned w = blockIdx.x * kWarpsPerBlock + wib, R = static_cast<unsigned>(s.R);
    if (w >= static_cast<unsigned>(s.B * s.Hkv) * R) return;
    const unsigned bg = w < R ? 0u : w / R;
    const int r = static_cast<int>(w - bg * R), b = s.B == 1 ? 0 : static_cast<int>(bg) / s.Hkv, g = static_cast<int>(bg) - b * s.Hkv;
    int32_t* sel = a.sel + ((static_cast<long long>(b) * s.Hkv + g) * s.R + r) * s.K;
    const int pos = row_position(a, b, r);
    if (pos < 0) {
        if (lane == 0) set_status(a.status, kDevBadIndex);
        for (int t = lane; t < s.K; t += 32) sel[t] = -1;
        return;
    }
    const int ncand = left_chunks(s, pos);
    if (ncand <= s.K) {                       // nothing to choose
        for (int t = lane; t < s.K; t += 32) sel[t] = t < ncand ? t : -1;
        return;
    }
    const int d = Quad<T, D, X>::dim(s.d), G = s.G, k8 = lane >> 2, at = (lane & 3) * Quad<T, D, X>::kE;
    const T* q = static_cast<const T*>(a.q_route);       // selection scores use the routing query
    const T* lm = static_cast<const T*>(a.lm);

    unsigned long long lst[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) lst[j] = 0ull;
    unsigned long long thr = 0ull;
    for (int base = 0; base < ncand; base += 32) {
        float u[4];                            // octet o: chunk base + 8 o + k8 (the same value in the quad's lanes)
#pragma unroll
        for (int o = 0; o < 4; ++o) u[o] = -INFINITY;
        for (int rr = 0; rr < G; ++rr) {
            Quad<T, D, X> qr;
            qr.load(q + ((static_cast<long long>(b) * s.Hq + g * G + rr) * s.R + r) * d + at, d);
            const int hl = (s.Hl == s.Hq) ? (g * G + rr) : g;
            const long long lrow = (static_cast<long long>(b) * s.Hl + hl) * s.C;
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                if (base + o * 8 >= ncand) break;
                const int c = min(base + o * 8 + k8, ncand - 1);
                Quad<T, D, X> x;
                x.load(lm + (lrow + c) * d + at, d);
                float sc = x.dot(qr) * s.scale;
                if (a.bias) sc += a.bias[lrow + c];
                u[o] = fmaxf(u[o], sc);
            }
        }
        // lane l: chunk base + l
        float mine = -INFINITY;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const float v = __shfl_sync(kFullMask, u[o], (lane & 7) * 4);
            if ((lane >> 3) == o) mine = v;
        }
        const unsigned long long key = base + lane < ncand ? select_key(mine, base + lane) : 0ull;
        unsigned pass = __ballot_sync(kFullMask, key > thr);
        if (__popc(pass) > 4) {
            list_merge<NR>(lst, key, s.K, lane);
            thr = __shfl_sync(kFullMask, lst[(s.K - 1) >> 5], (s.K - 1) & 31);
            pass = 0u;
        }
        while (pass) {
            const int src = __ffs(pass) - 1;
            pass &= pass - 1;
            const unsigned long long x = __shfl_sync(kFullMask, key, src);
            if (x > thr) {
                list_insert<NR>(lst, x, s.K, lane);
                thr = __shfl_sync(kFullMask, lst[(s.K - 1) >> 5], (s.K - 1) & 31);
            }
        }
    }

    // emit ascending chunk ids: rank of an id = number of selected ids below it (all K places are taken)
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const int mine = key_chunk(lst[j]);
        int rank = 0;
#pragma unroll
        for (int j2 = 0; j2 < NR; ++j2) {
            const int ids = key_chunk(lst[j2]);
            for (int l = 0; l < min(32, s.K - j2 * 32); ++l) rank += __shfl_sync(kFullMask, ids, l) < mine ? 1 : 0;
        }
        if (j * 32 + lane < s.K) sel[rank] = mine;
    }
}

// Scores of 64 keys from `base` on: octet o of the result holds key base + 8 o + lane / 4 (the same value in the quad's
// lanes), -inf from `hi` on.  k: this lane's piece of row 0.
template <typename T, int D, bool X>
__device__ __forceinline__ void score_64(const Quad<T, D, X>& q, const T* k, int base, int hi, int d, float scale, int k8, float (&sc)[8]) {
    if (base + 64 <= hi) {
        const T* row = k + static_cast<long long>(base + k8) * d;
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            Quad<T, D, X> x;
            x.load(row + static_cast<long long>(8 * o) * d, d);
            sc[o] = x.dot(q) * scale;
        }
    } else {
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            const int j = base + o * 8 + k8;
            sc[o] = -INFINITY;
            if (base + o * 8 < hi) {
                Quad<T, D, X> x;
                x.load(k + static_cast<long long>(min(j, hi - 1)) * d, d);
                const float v = x.dot(q) * scale;
                if (j < hi) sc[o] = v;
            }
        }
    }
}
__device__ __forceinline__ float octets_max(const float (&v)[8]) {
    float m = v[0];
#pragma unroll
    for (int o = 1; o < 8; ++o) m = fmaxf(m, v[o]);
#pragma unroll
    for (int x = 4; x < 32; x <<= 1) m = fmaxf(m, __shfl_xor_sync(kFullMask, m, x));
    return m;
}
__device__ __forceinline__ float octets_sum(const float (&v)[8]) {
    float m = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
#pragma unroll
    for (int x = 4; x < 32; x <<= 1) m += __shfl_xor_sync(kFullMask, m, x);
    return m;
}

// Per-chunk attention, local attention and fusion (Eq. HiLS weights; App. C per-head weights).  One CTA per (b, h, r);
// its warps take the row's items in turn: pieces of 64 tokens of the local window (their masses are exact, so mixing
// by the masses reproduces the window's single softmax), then the selected chunks.  The sums over the keys stay spread
// over the quads (a quad adds up its own keys) until the row is complete.
constexpr int kAttWarps = 8;
template <typename T, int D, bool X>
__global__ void __launch_bounds__(kAttWarps * 32, D <= 64 ? 3 : 1)
generic_attend_kernel(const GArgs a) {
    using Q = Quad<T, D, X>;
    __shared__ float part[kAttWarps][D];
    __shared__ float part_m[kAttWarps], part_d[kAttWarps];
    pdl_wait();
    const Shape& s = a.s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned orow = blockIdx.x;                           // (b Hq + h) R + r
    const int r = static_cast<int>(orow % static_cast<unsigned>(s.R));
    const int bh = static_cast<int>(orow / static_cast<unsigned>(s.R));
    const int h = bh % s.Hq, b = bh / s.Hq;
    const int g = h / s.G, d = Q::dim(s.d);
    T* out = static_cast<T*>(a.out) + static_cast<long long>(orow) * d;
    const int pos = row_position(a, b, r);
    if (pos < 0) {
        for (int t = threadIdx.x; t < d; t += blockDim.x) out[t] = from_f32<T>(0.f);
        if (threadIdx.x == 0) a.lse[orow] = 0.f;
        return;
    }
    const int lo = local_lo(pos, s.W, s.S);
    const int ncand = lo / s.S;
    const int k8 = lane >> 2, at = (lane & 3) * Q::kE;
    Q q;
    q.load(static_cast<const T*>(a.q) + static_cast<long long>(orow) * d + at, d);

    const T* kg = static_cast<const T*>(a.k) + (static_cast<long long>(b) * s.Hkv + g) * s.T * d + at;
    const T* vg = static_cast<const T*>(a.v) + (static_cast<long long>(b) * s.Hkv + g) * s.T * d + at;
    const int hl = (s.Hl == s.Hq) ? h : g;
    const long long lrow = (static_cast<long long>(b) * s.Hl + hl) * s.C;
    const int32_t* sel = a.sel + ((static_cast<long long>(b) * s.Hkv + g) * s.R + r) * s.K;

    const int n_loc = (pos - lo) / 64 + 1, n_items = n_loc + min(s.K, ncand);
    float Mx = kLowestLogit, Dn = 0.f;
    Q acc;
    acc.fill(0.f);
    for (int it = warp; it < n_items; it += nw) {
        int k0, k1;
        float lam = 0.f;
        if (it < n_loc) {
            k0 = lo + it * 64;
            k1 = min(pos + 1, k0 + 64);
        } else {
            const int c = sel[it - n_loc];
            if (c < 0 || c >= ncand) {              // never produced by the selection kernel
                if (lane == 0) set_status(a.status, kDevBadIndex);
                continue;
            }
            k0 = c * s.S;
            k1 = k0 + s.S;
            Q x, y;
            x.load(static_cast<const T*>(a.q_route) + static_cast<long long>(orow) * d + at, d);
            y.load(static_cast<const T*>(a.lm) + (lrow + c) * d + at, d);
            lam = x.dot(y) * s.scale + (a.bias ? a.bias[lrow + c] : 0.f);
        }
        float sc[8];
        score_64<T, D, X>(q, kg, k0, k1, d, s.scale, k8, sc);
        float m = octets_max(sc);
        if (k1 - k0 > 64)                          // chunks of more than 64 tokens: the maximum over the whole chunk first
            for (int base = k0 + 64; base < k1; base += 64) {
                float sx[8];
                score_64<T, D, X>(q, kg, base, k1, d, s.scale, k8, sx);
                m = fmaxf(m, octets_max(sx));
            }
#pragma unroll
        for (int o = 0; o < 8; ++o) sc[o] = __expf(sc[o] - m);
        float Z = octets_sum(sc);
        if (k1 - k0 > 64)
            for (int base = k0 + 64; base < k1; base += 64) {
                float sx[8];
                score_64<T, D, X>(q, kg, base, k1, d, s.scale, k8, sx);
#pragma unroll
                for (int o = 0; o < 8; ++o) sx[o] = __expf(sx[o] - m);
                Z += octets_sum(sx);
            }
        if (it < n_loc) lam = m + __logf(Z);
        const float Mn = fmaxf(Mx, lam);
        const float c_old = __expf(Mx - Mn), c_new = __expf(lam - Mn), w = c_new / Z;
        Dn = Dn * c_old + c_new;
        Mx = Mn;
        acc.scale_by(c_old);
        for (int base = k0;;) {
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                if (base + o * 8 >= k1) break;
                Q x;
                x.load(vg + static_cast<long long>(min(base + o * 8 + k8, k1 - 1)) * d, d);
                acc.add_scaled(sc[o] * w, x);
            }
            base += 64;
            if (base >= k1) break;
            score_64<T, D, X>(q, kg, base, k1, d, s.scale, k8, sc);
#pragma unroll
            for (int o = 0; o < 8; ++o) sc[o] = __expf(sc[o] - m);
        }
    }
    // the quads of the warp, then the warps (fixed order: deterministic)
#pragma unroll
    for (int i = 0; i < Q::kPl; ++i)
#pragma unroll
        for (int e = 0; e < Q::kE; ++e) {
            float v = acc.x[i][e];
#pragma unroll
            for (int x = 4; x < 32; x <<= 1) v += __shfl_xor_sync(kFullMask, v, x);
            acc.x[i][e] = v;
        }
    if (k8 == 0) {
#pragma unroll
        for (int i = 0; i < Q::kPl; ++i)
#pragma unroll
            for (int e = 0; e < Q::kE; ++e) part[warp][4 * Q::kE * i + at + e] = acc.x[i][e];
    }
    if (lane == 0) { part_m[warp] = Mx; part_d[warp] = Dn; }
    __syncthreads();
    float M = -INFINITY, den = 0.f;
    for (int w = 0; w < nw; ++w) M = fmaxf(M, part_m[w]);
    for (int w = 0; w < nw; ++w) den += part_d[w] * __expf(part_m[w] - M);
    for (int t = threadIdx.x; t < d; t += blockDim.x) {
        float v = 0.f;
        for (int w = 0; w < nw; ++w) v = fmaf(part[w][t], __expf(part_m[w] - M), v);
        out[t] = from_f32<T>(v / den);
    }
    if (threadIdx.x == 0) a.lse[orow] = M + __logf(den);
}

// ---- fp32 prefill on small shapes: chunk-major ------------------------------------------------------------------
// The row kernel above reads (K + 1) chunks per row, mostly from L2 (61 % of its requests on 2048 tokens, d = 64, K = 4;
// 38 us).  Here a CTA takes one chunk of one KV head and the tokens of a block that attend it: it looks their selections through,
// keeps K and V in shared memory and scores four or eight (token, head) rows at a time per warp (lane = key, then lane = dimension),
// so that a K or V value read from shared memory meets that many rows.  Partial outputs and masses per (row, slot) go through
// global memory to generic_fuse_kernel.
// Bound: shared-memory reads while all warps score (with eight rows as many cycles as the packed FMAs take, with four 1.5 times
// as many), latencies at both ends on small shapes.  The blocks are longer on larger shapes (launch_chunk_major): with blocks of 32
// tokens of one head the CTAs mostly loaded K and V (64 KB for six rows at 3072 tokens, d = 128, K = 4).
constexpr int kRowBlockMax = 128;

// Slots of a row: the selected chunks 0 .. K - 1, then the chunks of its local window.
__host__ __device__ inline int chunk_slots(const Shape& s) { return s.K + div_chunk(s, s.W + s.S - 2) + 1; }

// Chunks up to the last token of block r of rb tokens.
__host__ __device__ inline int block_chunks(const Shape& s, int rb, int r) { return div_chunk(s, s.pos0 + (s.R < (r + 1) * rb ? s.R : (r + 1) * rb) - 1) + 1; }

template <int D, int NW>
struct ChunkSmem {
    alignas(16) float k[64][D + 4];            // (padded: eight lanes reading the same piece of eight rows miss each other's banks)
    alignas(16) float v[64][D];
    union Warp {
        float q[NW][D];
        float4 p[64][NW / 2 + 1];                       // probabilities of a warp's rows per key, each twice (pairs of a packed multiply; padded)
    };
    alignas(16) Warp w[NW];
    int row[kRowBlockMax];                     // tokens (of the block) that attend the chunk and the slot they hold it in
    int slot[kRowBlockMax];
    int cnt[NW];
};

template <int D, int NW, int NR>
__device__ __forceinline__ void fetch_rows(const GArgs& a, const ChunkSmem<D, NW>& sm, int b, int h0, int nh, int n, int e0, float (&qv)[NR][D / 32]) {
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const int x = min(e0 + i, n * nh - 1), e = nh == 1 ? x : x / nh;
        const long long row = (static_cast<long long>(b) * a.s.Hq + h0 + (x - e * nh)) * a.s.R + sm.row[e];
#pragma unroll
        for (int y = 0; y < D / 32; ++y) qv[i][y] = static_cast<const float*>(a.q)[row * D + (threadIdx.x & 31) + 32 * y];
    }
}

// Rows (token, head) e0 .. e0 + NR - 1 of the n tokens x nh heads from h0 on (of KV head g), by one warp.  qv: their queries with four rows
// at a time (fetch_rows), and on return those of the rows from e0 + step on.
template <int D, int NW, int NR>
__device__ __forceinline__ void chunk_rows(const GArgs& a, ChunkSmem<D, NW>& sm, int c, int b, int g, int h0, int nh, int n, int e0, int step, float (&qv)[NR][D / 32], const float (&lmv)[D / 32],
                                           float* part, float* lam) {
    constexpr int kV = D / 32;                 // dimensions per lane in the value pass
    const Shape& s = a.s;
    const int lane = threadIdx.x & 31, NS = chunk_slots(s);
    typename ChunkSmem<D, NW>::Warp& w = sm.w[threadIdx.x >> 5];
    const bool own_lm = s.Hl == s.Hq && s.G > 1;                              // a landmark row per head
    long long orow[NR];                                                       // row of q
    int lim[NR], slot[NR], head[NR];
    float lm[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const int x = min(e0 + i, n * nh - 1), e = nh == 1 ? x : x / nh, r = sm.row[e];
        head[i] = h0 + (x - e * nh);
        orow[i] = (static_cast<long long>(b) * s.Hq + head[i]) * s.R + r;
        slot[i] = sm.slot[e];
        lim[i] = slot[i] < s.K ? s.S - 1 : min(s.S - 1, s.pos0 + r - c * s.S);
    }
    {
        if (NR > 4) fetch_rows<D, NW, NR>(a, sm, b, h0, nh, n, e0, qv);
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            lm[i] = 0.f;
            const float* lr = static_cast<const float*>(a.lm) + ((static_cast<long long>(b) * s.Hl + head[i]) * s.C + c) * D;
#pragma unroll
            for (int x = 0; x < kV; ++x) {
                w.q[i][lane + 32 * x] = qv[i][x];
                const float rv = a.q_route == a.q ? qv[i][x] : static_cast<const float*>(a.q_route)[orow[i] * D + lane + 32 * x];
                lm[i] = fmaf(rv, own_lm && c < s.C ? lr[lane + 32 * x] : lmv[x], lm[i]);
            }
        }
    }
    __syncwarp();
    if (NR == 4 && e0 + step < n * nh) fetch_rows<D, NW, NR>(a, sm, b, h0, nh, n, e0 + step, qv);
    // two dimensions per instruction: a pair's halves are added at the end
    float2 a0[NR], a1[NR];                                                    // keys lane, lane + 32
#pragma unroll
    for (int i = 0; i < NR; ++i) a0[i] = a1[i] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int x = 0; x < D; x += 4) {
        const float4 k0 = *reinterpret_cast<const float4*>(&sm.k[lane][x]), k1 = *reinterpret_cast<const float4*>(&sm.k[lane + 32][x]);
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const float4 qv = *reinterpret_cast<const float4*>(&w.q[i][x]);
            const float2 ql = make_float2(qv.x, qv.y), qh = make_float2(qv.z, qv.w);
            a0[i] = __ffma2_rn(ql, make_float2(k0.x, k0.y), a0[i]);
            a1[i] = __ffma2_rn(ql, make_float2(k1.x, k1.y), a1[i]);
            a0[i] = __ffma2_rn(qh, make_float2(k0.z, k0.w), a0[i]);
            a1[i] = __ffma2_rn(qh, make_float2(k1.z, k1.w), a1[i]);
        }
    }
    float mx[NR], z[NR], s0[NR], s1[NR];
    __syncwarp();                                                             // (the probabilities overwrite the queries)
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        s0[i] = lane <= lim[i] ? (a0[i].x + a0[i].y) * s.scale : -INFINITY;
        s1[i] = lane + 32 <= lim[i] ? (a1[i].x + a1[i].y) * s.scale : -INFINITY;
        mx[i] = fmaxf(s0[i], s1[i]);
    }
    // (the rows' reductions side by side: one after the other their shuffles would wait for one another)
#pragma unroll
    for (int x = 16; x > 0; x >>= 1)
#pragma unroll
        for (int i = 0; i < NR; ++i) mx[i] = fmaxf(mx[i], __shfl_xor_sync(kFullMask, mx[i], x));
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        s0[i] = __expf(s0[i] - mx[i]);
        s1[i] = __expf(s1[i] - mx[i]);
        z[i] = s0[i] + s1[i];
    }
#pragma unroll
    for (int x = 16; x > 0; x >>= 1)
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            z[i] += __shfl_xor_sync(kFullMask, z[i], x);
            lm[i] += __shfl_xor_sync(kFullMask, lm[i], x);
        }
#pragma unroll
    for (int i = 0; i < NR; i += 2) {
        w.p[lane][i / 2] = make_float4(s0[i], s0[i], s0[i + 1], s0[i + 1]);
        w.p[lane + 32][i / 2] = make_float4(s1[i], s1[i], s1[i + 1], s1[i + 1]);
    }
    __syncwarp();
    float2 o[NR][kV / 2];
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
        for (int x = 0; x < kV / 2; ++x) o[i][x] = make_float2(0.f, 0.f);
#pragma unroll (NR == 4 ? 8 : 4)
    for (int j = 0; j < 64; ++j) {
        float4 p[NR / 2];
#pragma unroll
        for (int i = 0; i < NR / 2; ++i) p[i] = w.p[j][i];
#pragma unroll
        for (int x = 0; x < kV / 2; ++x) {
            const float2 v = *reinterpret_cast<const float2*>(&sm.v[j][2 * lane + 64 * x]);
#pragma unroll
            for (int i = 0; i < NR; i += 2) {
                o[i][x] = __ffma2_rn(make_float2(p[i / 2].x, p[i / 2].y), v, o[i][x]);
                o[i + 1][x] = __ffma2_rn(make_float2(p[i / 2].z, p[i / 2].w), v, o[i + 1][x]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        if (e0 + i >= n * nh) break;
        const long long at = orow[i] * NS + slot[i];
        const float zi = 1.f / z[i];
#pragma unroll
        for (int x = 0; x < kV / 2; ++x)
            *reinterpret_cast<float2*>(part + at * D + 2 * lane + 64 * x) = make_float2(o[i][x].x * zi, o[i][x].y * zi);
        if (lane == 0) {
            const int hl = s.Hl == s.Hq ? head[i] : g;
            lam[at] = slot[i] < s.K ? lm[i] * s.scale + (a.bias ? a.bias[(static_cast<long long>(b) * s.Hl + hl) * s.C + c] : 0.f)
                                    : mx[i] + __logf(z[i]);
        }
    }
    __syncwarp();
}

// NW: warps per CTA and most rows of a warp at a time, row_block: tokens (nb blocks), nh: query heads (of one KV head), mid_first: whether
// the blocks are walked from the middle ones on (see chunk_form)
template <int D, int NW>
__global__ void __launch_bounds__(NW * 32, 16 / NW)
generic_chunk_kernel(const GArgs a, int row_block, int nb, int nh, int mid_first, float* part, float* lam) {
    extern __shared__ uint8_t chunk_raw[];
    ChunkSmem<D, NW>& sm = *reinterpret_cast<ChunkSmem<D, NW>*>(chunk_raw);
    const Shape& s = a.s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // two blocks of tokens, as far from the first one as from the last, share a row of CTAs, one per chunk up to their last tokens: from the
    // ends on with the late one first, or from the middle on with the early one, whose tokens attend most of their chunks, first
    const int y = mid_first ? gridDim.y - 1 - blockIdx.y : nb - 1 - blockIdx.y, n_y = block_chunks(s, row_block, y);
    const bool other = static_cast<int>(blockIdx.x) >= n_y;
    const int blk = other ? nb - 1 - y : y, c = other ? blockIdx.x - n_y : blockIdx.x;
    if (other && (blk == y || c >= block_chunks(s, row_block, blk))) return;
    int b = 0, g = blockIdx.z, h0 = 0;                                      // z: (sequence, KV head, nh of its query heads)
    if (nh < s.G) {
        const int per = s.G / nh;
        g = blockIdx.z / per;
        h0 = (blockIdx.z - g * per) * nh;
    }
    if (s.B > 1) {
        b = g / s.Hkv;
        g -= b * s.Hkv;
    }
    h0 += g * s.G;
    const int r0 = blk * row_block;
    const float* kc = static_cast<const float*>(a.k) + ((static_cast<long long>(b) * s.Hkv + g) * s.T + static_cast<long long>(c) * s.S) * D;
    const float* vc = static_cast<const float*>(a.v) + (kc - static_cast<const float*>(a.k));
    // rows of the chunk up to the call's last token: the ones after it may hold anything, and 0 x NaN is NaN
    const int rows_k = min(s.S, s.pos0 + s.R - c * s.S);
    for (int x = tid; x < rows_k * (D / 4); x += blockDim.x)
        cp_async16(smem_u32(&sm.k[x / (D / 4)][(x % (D / 4)) * 4]), kc + x * 4);
    for (int x = tid; x < rows_k * (D / 4); x += blockDim.x)
        cp_async16(smem_u32(&sm.v[x / (D / 4)][(x % (D / 4)) * 4]), vc + x * 4);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int x = rows_k * D + tid; x < 64 * D; x += blockDim.x) { sm.k[x / D][x % D] = 0.f; sm.v[x / D][x % D] = 0.f; }
    float lmv[D / 32];                          // the chunk's landmark (with one per head: not used)
#pragma unroll
    for (int x = 0; x < D / 32; ++x)
        lmv[x] = c < s.C ? static_cast<const float*>(a.lm)[((static_cast<long long>(b) * s.Hl + (s.Hl == s.Hq ? g * s.G : g)) * s.C + c) * D + lane + 32 * x] : 0.f;
    pdl_wait();                                 // the selection
    int slot = -1;
    {
        const int r = r0 + tid, pos = s.pos0 + r;
        if (tid < row_block && r < s.R && c * s.S <= pos) {
            const int lc = left_chunks(s, pos);
            if (c >= lc) {
                slot = s.K + c - lc;
            } else {
                const int32_t* sel = a.sel + ((static_cast<long long>(b) * s.Hkv + g) * s.R + r) * s.K;
                for (int t = 0; t < s.K; ++t) if (sel[t] == c) slot = t;
            }
        }
        const unsigned vote = __ballot_sync(kFullMask, slot >= 0);
        if (lane == 0) sm.cnt[warp] = __popc(vote);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        int at = __popc(vote & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) at += sm.cnt[w];
        if (slot >= 0) { sm.row[at] = r; sm.slot[at] = slot; }
    }
    int n = 0;
    for (int w = 0; w < NW; ++w) n += sm.cnt[w];
    __syncthreads();
    const int rows = n * nh;
    if (NW == 8 && rows > NW * 4) {
        float qv[8][D / 32];
        for (int e0 = warp * 8; e0 < rows; e0 += NW * 8) chunk_rows<D, NW, 8>(a, sm, c, b, g, h0, nh, n, e0, NW * 8, qv, lmv, part, lam);
    } else if (warp * 4 < rows) {
        float qv[4][D / 32];
        fetch_rows<D, NW, 4>(a, sm, b, h0, nh, n, warp * 4, qv);
        for (int e0 = warp * 4; e0 < rows; e0 += NW * 4) chunk_rows<D, NW, 4>(a, sm, c, b, g, h0, nh, n, e0, NW * 4, qv, lmv, part, lam);
    }
}

// Mix of a row's slots (Eq. HiLS weights): one warp per (b, h, r).
template <int D>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
generic_fuse_kernel(const GArgs a, const float* part, const float* lam) {
    constexpr int kV = D / 32;
    pdl_wait();
    const Shape& s = a.s;
    const int lane = threadIdx.x & 31;
    const unsigned row = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5), R = static_cast<unsigned>(s.R);
    if (row >= static_cast<unsigned>(s.B * s.Hq) * R) return;
    const int pos = s.pos0 + static_cast<int>(row < R ? row : row % R), lc = left_chunks(s, pos);
    const long long orow = row;
    const int NS = chunk_slots(s), nsel = min(s.K, lc), nl = div_chunk(s, pos) - lc + 1;
    const float* lr = lam + orow * NS;
    auto slot_of = [&](int i) { return i < nsel ? i : s.K + (i - nsel); };
    float M = -INFINITY;
    for (int i = lane; i < nsel + nl; i += 32) M = fmaxf(M, lr[slot_of(i)]);
    M = warp_max(M);
    float den = 0.f, o[kV];
#pragma unroll
    for (int x = 0; x < kV; ++x) o[x] = 0.f;
#pragma unroll 4
    for (int i = 0; i < nsel + nl; ++i) {
        const int t = slot_of(i);
        const float w = __expf(lr[t] - M);
        const float* src = part + (orow * NS + t) * D + lane;
        den += w;
#pragma unroll
        for (int x = 0; x < kV; ++x) o[x] = fmaf(w, src[32 * x], o[x]);
    }
    float* out = static_cast<float*>(a.out) + orow * D + lane;
#pragma unroll
    for (int x = 0; x < kV; ++x) out[32 * x] = o[x] / den;
    if (lane == 0) a.lse[orow] = M + __logf(den);
}

// The chunk-major kernels apply while the partial outputs stay small and looking every row's selection through once per
// visible chunk stays cheap beside the attention itself (both hold up to about 4K tokens).
bool chunk_major(const Shape& s, int dtype) {
    if (dtype != HILS_F32 || s.is_decode || s.S > 64 || (s.d != 64 && s.d != 128)) return false;
    const long long rows = static_cast<long long>(s.B) * s.Hq * s.R, chunks = (s.pos0 + s.R + s.S - 1) / s.S;
    return chunks <= 65535 && static_cast<long long>(s.B) * s.Hq <= 65535 && rows * chunk_slots(s) * s.d * 4 <= (256ll << 20) &&
           rows * chunks * s.K * 4 <= (256ll << 20);
}
size_t chunk_lam_offset(const Shape& s) {
    return (static_cast<size_t>(s.B) * s.Hq * s.R * chunk_slots(s) * s.d * sizeof(float) + 255) / 256 * 256;
}

// (block, chunk) pairs with blocks of rb tokens, over all KV heads
long long chunk_ctas(const Shape& s, int rb) {
    long long n = 0;
    for (int r = 0; r * rb < s.R; ++r) n += block_chunks(s, rb, r);
    return n * s.B * s.Hkv;
}

// Three block sizes: 32 tokens of one query head (most CTAs, least work each), 64 tokens of one head, 128 tokens with all query heads
// of the KV head (a K or V value is fetched for the most rows); four warps at d = 64, eight at d = 128.  The lines lie where the
// counts of 32-token CTAs below cross, K = 8, us for the call (32 / 64 / 128 tokens):
//   d = 128: 841 tokens, 4 heads (2 KV heads) 48 / 54 / 67; 2048, one head 51 / 47 / 54; 2048, 4 heads (2) 149 / 128 / 142;
//            3000, 2 heads (1) 141 / 112 / 110; 4096, 4 heads (2) 448 / 316 / 259
//   d = 64:  8 x 841, one head 55 / 62 / 65; 2048, 2 heads (1) 51 / 52 / 60; 2048, 4 heads (2) 87 / 82 / 90; 3 x 2048, 4 heads (2)
//            227 / 203 / 221; 3 x 3300, 4 heads (2) 459 / 371 / 346
// (with four warps for 32 tokens everywhere and eight for 128, one line between them: 56, 55, 142, 110, 260; 66, 51, 101, 227, 380)
// Where a few of the 32-token CTAs are left over from the first that are resident (four per SM at d = 64, two at 128), the blocks are walked
// from the middle on, which leaves the last blocks' chunks, with the fewest rows, for the end; elsewhere from the ends on (us, one head,
// d = 64, from the middle / from the ends: 1612 tokens, K = 8, 1.14 times the resident CTAs, 29.2 / 31.4; 1800, 1.42 times, 31.0 / 32.6; 2048
// tokens, K = 4, 1.78 times, 29.5 / 28.1).
struct ChunkForm { int tokens, heads, warps, mid_first; };        // per CTA: tokens, query heads of a KV head, warps
ChunkForm chunk_form(const Shape& s) {
    const long long ctas = chunk_ctas(s, 32), heads = ctas * s.G, sms = sm_count();
    const int warps = s.d == 64 ? 4 : 8;
    if (ctas >= (s.d == 64 ? 60 : 15) * sms) return {kRowBlockMax, s.G, warps, 0};
    if (heads >= (s.d == 64 ? 24 : 7) * sms) return {64, 1, warps, 0};
    return {32, 1, warps, 10 * heads <= 16 * (16 / warps) * sms ? 1 : 0};
}

template <int D, int NW>
int launch_chunk_kernel(const GArgs& a, int rb, int nh, int mid_first, float* part, float* lam, cudaStream_t stream) {
    const Shape& s = a.s;
    static PerDeviceOnce once;
    if (once.pending()) {
        if (cudaFuncSetAttribute(generic_chunk_kernel<D, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(ChunkSmem<D, NW>)) != cudaSuccess)
            return HILS_ERR_CUDA;
        once.done();
    }
    const int nb = (s.R + rb - 1) / rb;
    int width = 0;
    for (int y = 0; y < (nb + 1) / 2; ++y) {
        const int w = block_chunks(s, rb, nb - 1 - y) + (y < nb - 1 - y ? block_chunks(s, rb, y) : 0);
        width = w > width ? w : width;
    }
    return launch_pdl(generic_chunk_kernel<D, NW>, dim3(static_cast<unsigned>(width), static_cast<unsigned>((nb + 1) / 2), static_cast<unsigned>(s.B * s.Hq / nh)), dim3(NW * 32),
                      sizeof(ChunkSmem<D, NW>), stream, a, rb, nb, nh, mid_first, part, lam) == cudaSuccess ? 0 : HILS_ERR_CUDA;
}

template <int D>
int launch_chunk_major(const GArgs& a, void* scratch, cudaStream_t stream) {
    const Shape& s = a.s;
    float* part = static_cast<float*>(scratch);
    float* lam = reinterpret_cast<float*>(static_cast<char*>(scratch) + chunk_lam_offset(s));
    const long long rows = static_cast<long long>(s.B) * s.Hq * s.R;
    const ChunkForm f = chunk_form(s);
    if (launch_chunk_kernel<D, D == 64 ? 4 : 8>(a, f.tokens, f.heads, f.mid_first, part, lam, stream) != 0) return HILS_ERR_CUDA;
    trace_mark("generic_attend", stream);
    if (launch_pdl(generic_fuse_kernel<D>, dim3(static_cast<unsigned>((rows + kWarpsPerBlock - 1) / kWarpsPerBlock)),
                   dim3(kWarpsPerBlock * 32), 0, stream, a, static_cast<const float*>(part), static_cast<const float*>(lam)) != cudaSuccess)
        return HILS_ERR_CUDA;
    trace_mark("generic_fuse", stream);
    return 3;
}

template <typename T, int D, bool X>
int launch_dim(const GArgs& a, void* scratch, cudaStream_t stream) {
    const Shape& s = a.s;
    const long long sel_warps = static_cast<long long>(s.B) * s.Hkv * s.R;
    const long long rows = static_cast<long long>(s.B) * s.Hq * s.R;
    if (rows > 0x7fffffffll) return HILS_ERR_UNSUPPORTED;
    const unsigned sel_blocks = static_cast<unsigned>((sel_warps + kWarpsPerBlock - 1) / kWarpsPerBlock);
    const int nr = (s.K + 31) / 32;
    if (nr <= 1) generic_select_kernel<T, D, X, 1><<<sel_blocks, kWarpsPerBlock * 32, 0, stream>>>(a);
    else if (nr == 2) generic_select_kernel<T, D, X, 2><<<sel_blocks, kWarpsPerBlock * 32, 0, stream>>>(a);
    else generic_select_kernel<T, D, X, 4><<<sel_blocks, kWarpsPerBlock * 32, 0, stream>>>(a);
    if (cudaGetLastError() != cudaSuccess) return HILS_ERR_CUDA;
    trace_mark("generic_select", stream);
    if (scratch) return s.d == 64 ? launch_chunk_major<64>(a, scratch, stream) : launch_chunk_major<128>(a, scratch, stream);
    // a warp per item of the row, at most eight
    const long long items = static_cast<long long>(s.K) + (s.W + s.S - 2) / 64 + 1;
    const unsigned warps = static_cast<unsigned>(items < kAttWarps ? items : kAttWarps);
    if (launch_pdl(generic_attend_kernel<T, D, X>, dim3(static_cast<unsigned>(rows)), dim3(warps * 32), 0, stream, a) != cudaSuccess)
        return HILS_ERR_CUDA;
    trace_mark("generic_attend", stream);
    return 2;
}

// (scratch: for the chunk-major kernels; none where they do not apply)
template <typename T>
int launch_typed(const GArgs& a, void* scratch, cudaStream_t stream) {
    if (a.s.d == 64) return launch_dim<T, 64, true>(a, scratch, stream);
    if (a.s.d == 128) return launch_dim<T, 128, true>(a, scratch, stream);
    if (a.s.d < 128) return launch_dim<T, 128, false>(a, scratch, stream);
    return launch_dim<T, 256, false>(a, scratch, stream);
}

}  // namespace

bool generic_supports(const Shape& s) {
    return s.d % 32 == 0 && s.d >= 32 && s.d <= 256 && s.K >= 1 && s.K <= 128 && s.G * s.d <= 2048 &&
           s.S >= 1;
}

size_t generic_scratch_bytes(const Shape& s, int dtype) {
    if (!chunk_major(s, dtype)) return 0;
    return chunk_lam_offset(s) + sizeof(float) * static_cast<size_t>(s.B) * s.Hq * s.R * chunk_slots(s);
}

void generic_chunk_form(const Shape& s, int dtype, int32_t* form) {
    if (!chunk_major(s, dtype)) return;
    const ChunkForm f = chunk_form(s);
    form[0] = f.tokens;
    form[1] = f.heads;
    form[2] = f.warps;
    form[3] = f.mid_first;
}

int launch_generic(const Shape& s, int dtype, const Tensors& t, cudaStream_t stream) {
    if (!generic_supports(s)) return HILS_ERR_UNSUPPORTED;
    GArgs a{s, t.q, t.q_route ? t.q_route : t.q, t.k, t.v, t.landmarks, t.bias, t.seq_lens, t.out, t.lse, t.sel_idx, t.status};
    // a workspace without room for the chunk-major kernels' partial outputs: the row kernel
    void* scratch = chunk_major(s, dtype) && t.scratch_bytes >= generic_scratch_bytes(s, dtype) ? t.scratch : nullptr;
    if (dtype == HILS_F32) return launch_typed<float>(a, scratch, stream);
    return launch_typed<__nv_bfloat16>(a, scratch, stream);
}

}  // namespace hils
