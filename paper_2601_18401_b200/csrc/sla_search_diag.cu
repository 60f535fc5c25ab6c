// Span-search for bf16, head_dim 128 and groups of 4, 8 or 16 query heads per KV head (Section "Span
// search": s_{i,t} = <Q_s(i), K(t)> over the anchors t_s = i + 1 - offset(s), then TopK), with the
// selection folded into the scoring loop.
//
// The fixed stride pattern makes the keys of one stride contiguous over consecutive queries: query
// i0 + j scores key t0 + j at stride s (Section "Span search": "the fixed stride pattern allows us to
// calculate the search scores in a more efficient manner").  A warp owns four consecutive query
// positions of one (batch, KV head).  Its routing queries -- 4 positions x 4 heads -- are the 16 rows
// of the A operand of an m16n8k16 tensor-core MMA and stay in registers for the whole row of strides;
// the 8 columns of the B operand are the keys of two strides for the four positions, fetched with
// plain 32-byte loads (every key row is needed by exactly one position per stride, so there is
// nothing to share through shared memory; K stays in L2).  Of the 16 x 8 products of an MMA the
// 4 x 4 x 2 diagonal blocks are scores -- exactly one per lane: lane (row group r8, quad index q)
// receives the score of (position 2(q&1) + (r8>>2), head r8&3) at stride s0 + (q>>1).  So every lane
// owns one (position, head) pair on every other stride and keeps that pair's running top-k itself:
//   - the K best values so far, sorted, in registers (a branch-free insertion of two min/max per slot);
//   - every score that beat the K-th best when it arrived is appended with its stride index to the
//     lane's list in shared memory -- the final selection is a subset of that list.  When a list runs
//     full, the warp's lanes drop the entries that have fallen below their K-th best since.
// At the end each lane sorts out the stride indices of its K best, the two lanes of a pair merge their
// lists through shuffles (larger score first, smaller stride index on ties) and write the slots.
// The dims are assigned to the MMA's k slots in a permuted order (identical for A and B, which leaves
// the dot product unchanged) so that each lane loads 32 contiguous bytes of a row and a quad a whole
// 128-byte line.
#include <limits.h>
#include <math_constants.h>

#include "sla_kernels.h"
#include "sla_topk.cuh"

namespace sla {

namespace {

using bf16 = __nv_bfloat16;
constexpr int kWarps = 8;
constexpr int kQW = 4;   // query positions per warp
constexpr int kG = 4;    // query heads per KV head

template <int K> struct ListCap { static constexpr int value = (2 * K + 8 + 3) / 4 * 4; };

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 32 bytes per lane in one load: the four lanes of a quad cover a whole 128-byte line of a row, so a warp's
// load touches eight full lines (with 16-byte loads it would touch the same eight lines for half the bytes)
struct Words8 { uint32_t w[8]; };
__device__ __forceinline__ Words8 ldg256(const void *p) {
    Words8 r;
    asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
                 : "l"(p));
    return r;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Descending order of (score, stride): larger score first, smaller stride index on ties.
__device__ __forceinline__ bool beats(float xa, int sa, float xb, int sb) { return xa > xb || (xa == xb && sa < sb); }

// Batcher's odd-even merge sort of K (a power of two) register-resident (score, stride) pairs, best first.
template <int K>
__device__ __forceinline__ void sort_pairs(float (&x)[K], int (&s)[K]) {
#pragma unroll
    for (int p = 1; p < K; p <<= 1)
#pragma unroll
        for (int k = p; k >= 1; k >>= 1)
#pragma unroll
            for (int a = 0; a < K; ++a) {
                // a is the upper element of a comparator (a, a + k) of this stage of the network
                const int j0 = k % p, b = a + k;
                if (a >= j0 && (a - j0) % (2 * k) < k && b < K && a / (2 * p) == b / (2 * p)) {
                    const bool sw = beats(x[b], s[b], x[a], s[a]);
                    const float xa = sw ? x[b] : x[a], xb = sw ? x[a] : x[b];
                    const int sa = sw ? s[b] : s[a], sb = sw ? s[a] : s[b];
                    x[a] = xa; x[b] = xb; s[a] = sa; s[b] = sb;
                }
            }
}

// The K best of this lane's and of lane ^ off's sorted lists, in both lanes: the j-th of one against the (K-1-j)-th of the
// other leaves them as a bitonic sequence, which log2 K rounds of half-cleaners sort.
template <int K>
__device__ __forceinline__ void merge_pairs(float (&x)[K], int (&s)[K], int off) {
    float px[K];
    int ps[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        px[j] = __shfl_xor_sync(0xffffffffu, x[j], off);
        ps[j] = __shfl_xor_sync(0xffffffffu, s[j], off);
    }
#pragma unroll
    for (int j = 0; j < K; ++j)
        if (beats(px[K - 1 - j], ps[K - 1 - j], x[j], s[j])) {
            x[j] = px[K - 1 - j];
            s[j] = ps[K - 1 - j];
        }
#pragma unroll
    for (int d = K / 2; d >= 1; d >>= 1)
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((j & d) == 0) {
                const bool sw = beats(x[j + d], s[j + d], x[j], s[j]);
                const float xa = sw ? x[j + d] : x[j], xb = sw ? x[j] : x[j + d];
                const int sa = sw ? s[j + d] : s[j], sb = sw ? s[j] : s[j + d];
                x[j] = xa; x[j + d] = xb; s[j] = sa; s[j + d] = sb;
            }
}

// A lane's running top-k: the K best values so far, sorted, in registers, and in shared memory (entry e at lx[32 e],
// ls[32 e]) every score with its stride index that beat the K-th best when it arrived.
template <int K>
struct RunningTop {
    static constexpr int CAP = ListCap<K>::value;
    float v[K];
    int cnt;
    float *lx;
    int *ls;
    __device__ __forceinline__ RunningTop(float *warp_lists, int lane)
        : cnt(0), lx(warp_lists + lane), ls(reinterpret_cast<int *>(warp_lists + CAP * 32) + lane) {
#pragma unroll
        for (int j = 0; j < K; ++j) v[j] = -CUDART_INF_F;
    }
    // Drops the list entries that can no longer be among the K best (all lanes, each its own list):
    // what is left are the entries above the K-th best value and the earliest of those equal to it,
    // at most K in all, still in stride order.
    __device__ __forceinline__ void compact() {
        const float vk = v[K - 1];
        int allow_eq = K;
#pragma unroll
        for (int j = 0; j < K; ++j) allow_eq -= v[j] > vk;
        int w = 0;
        for (int e0 = 0; e0 < cnt; e0 += 4) {   // four loads at a time: the list is as long as a multiple of four
            float x[4];
            int s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                x[u] = lx[32 * (e0 + u)];
                s[u] = ls[32 * (e0 + u)];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool eq = x[u] == vk;
                if (e0 + u < cnt && (x[u] > vk || (eq && allow_eq > 0))) {
                    allow_eq -= eq;
                    lx[32 * w] = x[u];
                    ls[32 * w] = s[u];
                    ++w;
                }
            }
        }
        cnt = w;
    }
    // Two new scores, sa < sb.  Each one that beats the K-th best so far goes to the list; the sorted values take
    // both in one pass: with hi >= lo the new j-th best is max(v[j], min(v[j-1], hi), min(v[j-2], lo)).
    __device__ __forceinline__ void offer2(int sa, float xa, int sb, float xb) {
        if (__any_sync(0xffffffffu, cnt >= CAP - 1)) compact();   // room for both scores
        const float vk = v[K - 1];
        if (xa > vk) {
            lx[32 * cnt] = xa;
            ls[32 * cnt] = sa;
            ++cnt;
        }
        if (xb > vk) {
            lx[32 * cnt] = xb;
            ls[32 * cnt] = sb;
            ++cnt;
        }
        const float hi = fmaxf(xa, xb), lo = fminf(xa, xb);
#pragma unroll
        for (int j = K - 1; j >= 2; --j) v[j] = max3(v[j], fminf(v[j - 1], hi), fminf(v[j - 2], lo));
        if (K >= 2) v[1] = max3(v[1], fminf(v[0], hi), lo);
        v[0] = fmaxf(v[0], hi);
    }
    // The K best with their stride indices, best first; absent entries are (-inf, INT_MAX).
    __device__ __forceinline__ void finish(float (&x)[K], int (&s)[K]) {
        compact();
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const bool on = j < cnt;
            x[j] = on ? lx[32 * j] : -CUDART_INF_F;
            s[j] = on ? ls[32 * j] : INT_MAX;
        }
        sort_pairs<K>(x, s);
    }
};

// The running lists take two scores at a time, neither of them NaN, and only those above -inf.  A warp that met an Inf or
// NaN among its scores selects again, a pass over the strides per slot: the largest score after the one taken last (smaller
// stride on ties); a NaN is no candidate, -inf comes after all others.
struct NextBest {
    unsigned taken = 0xffffffffu, key = 0u;   // order keys: of the score taken last; of the best after it (0: none)
    int at = -1, s = INT_MAX;                 // their strides
    __device__ __forceinline__ void offer(int sx, float x) {
        const unsigned kx = max(topk::order_key(x), 1u);
        if (x == x && (kx < taken || (kx == taken && sx > at)) && kx > key) { key = kx; s = sx; }
    }
    __device__ __forceinline__ void merge(int off) {
        const unsigned ok = __shfl_xor_sync(0xffffffffu, key, off);
        const int os = __shfl_xor_sync(0xffffffffu, s, off);
        if (ok > key || (ok == key && os < s)) { key = ok; s = os; }
    }
    __device__ __forceinline__ bool found() const { return s != INT_MAX; }
    __device__ __forceinline__ float score() const {
        return found() ? __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key) : -CUDART_INF_F;
    }
    __device__ __forceinline__ void take() { taken = key; at = s; key = 0u; s = INT_MAX; }
};

template <int K>
__global__ void __launch_bounds__(kWarps * 32, 2)
search_diag(const bf16 *__restrict__ q_s, const bf16 *__restrict__ k, Call c, int32_t *__restrict__ out_anchor,
            float *__restrict__ out_score) {
    extern __shared__ float smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r8 = lane >> 2, q = lane & 3;
    // the tiles with the most strides (the last positions) start first
    const long long r0 = ((long long)(gridDim.x - 1 - blockIdx.x) * kWarps + warp) * kQW;
    if (r0 >= c.Lq) return;
    const int bg = blockIdx.y, g = bg % c.Hkv, b = bg / c.Hkv;

    const long long last = c.Lq - 1;
    // ---- A operand: rows r8 and r8 + 8 = (position r8>>2, head r8&3) and (position 2 + (r8>>2), head r8&3)
    Words8 qa[2], qb[2];
    chain_wait();
    {
        const long long ra = r0 + (r8 >> 2) < last ? r0 + (r8 >> 2) : last;
        const long long rb = r0 + 2 + (r8 >> 2) < last ? r0 + 2 + (r8 >> 2) : last;
        const bf16 *base = q_s + b * c.q_sb + (long long)(g * kG + (r8 & 3)) * c.q_sh + 16 * q;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            qa[j] = ldg256(base + ra * c.q_st + 64 * j);
            qb[j] = ldg256(base + rb * c.q_st + 64 * j);
        }
    }
    // strides of the warp's positions: one integer square root per warp (quadratic pattern), the other
    // positions have as many strides or one more
    const int i0 = (int)(c.q_pos0 + r0);   // positions fit 31 bits
    const int n0 = n_strides(c, i0);
    auto n_at = [&](int i) -> int {
        if (c.off) return n_strides(c, i);
        return n0 + ((long long)(n0 + 1) * (n0 + 1) <= (long long)i + 1);
    };
    // ---- loader role: column r8 of the B operand = key of position jc at stride s0 + u_ld
    const int jc = r8 & 3, u_ld = r8 >> 2;
    const bool row_ld = r0 + jc <= last;
    const int i_ld = row_ld ? i0 + jc : (int)(c.q_pos0 + last);
    const int n_ld = row_ld ? n_at(i_ld) : 0;
    // ---- owner role: the score this lane receives
    const int jq = ((q & 1) << 1) | (r8 >> 2), hh = r8 & 3, u_own = q >> 1;
    const bool row_own = r0 + jq <= last;
    const int i_own = row_own ? i0 + jq : (int)(c.q_pos0 + last);
    const int n_own = row_own ? n_at(i_own) : 0;
    // Algorithm 1: anchors inside the local window are no candidates; t_s lies in W iff offset(s) <= w
    const int s_min = c.window > 0 ? window_strides(c) : 0;
    const bool full_group = r0 + kQW - 1 <= last;
    const int n_max = full_group ? n_at(i0 + kQW - 1) : n_at((int)(c.q_pos0 + last));
    const int n_all = full_group ? n0 : s_min;   // strides below n_all exist for every position of the warp

    const bf16 *kbase = k + b * c.kv_sb + g * c.kv_sh + 16 * q;
    const int kv_st = (int)c.kv_st;
    auto fetch = [&](int s0, Words8 (&kb)[2]) {
        const int s = s0 + u_ld;
        int t = i_ld + 1 - stride_offset(c, s < c.n_off || !c.off ? s : 0);
        if (s >= n_ld) t = i_ld;   // a valid row either way
        const bf16 *row = kbase + (long long)t * kv_st;
        kb[0] = ldg256(row);
        kb[1] = ldg256(row + 64);
    };

    RunningTop<K> top(smem + (size_t)warp * (2 * RunningTop<K>::CAP * 32), lane);
    // scores of one B tile (two strides): two independent accumulation chains, added at the end
    auto score = [&](const Words8 (&kb)[2]) -> float {
        float a0[4] = {0.f, 0.f, 0.f, 0.f}, a1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            mma_bf16_16816(a0, qa[0].w[2 * x], qb[0].w[2 * x], qa[0].w[2 * x + 1], qb[0].w[2 * x + 1], kb[0].w[2 * x], kb[0].w[2 * x + 1]);
            mma_bf16_16816(a1, qa[1].w[2 * x], qb[1].w[2 * x], qa[1].w[2 * x + 1], qb[1].w[2 * x + 1], kb[1].w[2 * x], kb[1].w[2 * x + 1]);
        }
        // the one score of this lane: row r8 (positions 0, 1) or r8 + 8 (positions 2, 3), column 2q + (r8>>2)
        const float lo = (r8 >> 2) ? a0[1] + a1[1] : a0[0] + a1[0], hi = (r8 >> 2) ? a0[3] + a1[3] : a0[2] + a1[2];
        return ((q & 1) ? hi : lo) * c.search_scale;
    };
    // two B tiles of two strides, each fetched again as soon as its scores are taken (32768 x 2 positions, K = 2 and
    // 16384 positions, K = 8: 1.2 to 1.5 % off search and attention together against fetch and use in one step)
    Words8 ka[2], kb[2];
    int s0 = s_min;
    float zero = 0.f;   // zero times the scores: NaN once one of them is not finite
    fetch(s0, ka);
    fetch(s0 + 2, kb);
    for (; s0 + 4 <= n_all; s0 += 4) {
        const float xa = score(ka);
        fetch(s0 + 4, ka);
        const float xb = score(kb);
        fetch(s0 + 6, kb);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s0 + u_own, xa, s0 + 2 + u_own, xb);
    }
    for (; s0 < n_max; s0 += 4) {
        float xa = score(ka), xb = score(kb);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        xa = s0 + u_own < n_own ? xa : -CUDART_INF_F;
        xb = s0 + 2 + u_own < n_own ? xb : -CUDART_INF_F;
        top.offer2(s0 + u_own, xa, s0 + 2 + u_own, xb);
        if (s0 + 4 < n_max) {
            fetch(s0 + 4, ka);
            fetch(s0 + 6, kb);
        }
    }

    const long long obase = ((((long long)b * c.Hq + g * kG + hh) * c.Lq) + r0 + jq) * c.top_k;
    if (__any_sync(0xffffffffu, zero != 0.f)) {
        NextBest next;
#pragma unroll 1
        for (int j = 0; j < c.top_k; ++j) {
#pragma unroll 1
            for (int s1 = s_min; s1 < n_max; s1 += 2) {
                fetch(s1, ka);
                const float x = score(ka);
                if (s1 + u_own < n_own) next.offer(s1 + u_own, x);
            }
            next.merge(2);
            if (row_own && u_own == 0) {
                out_anchor[obase + j] = next.found() ? i_own + 1 - stride_offset(c, next.s) : -1;
                out_score[obase + j] = next.score();
            }
            next.take();
        }
        return;
    }
    // ---- the lane's K best, merged with those of the lane that holds the pair's other strides (q differs in bit 1);
    // either of the two writes every other slot
    float ex[K];
    int es[K];
    top.finish(ex, es);
    merge_pairs<K>(ex, es, 2);
    if (!row_own) return;
#pragma unroll
    for (int j = 0; j < K; ++j)
        if ((j & 1) == u_own && j < c.top_k) {
            const bool on = es[j] != INT_MAX;
            out_anchor[obase + j] = on ? i_own + 1 - stride_offset(c, es[j]) : -1;
            out_score[obase + j] = on ? ex[j] : -CUDART_INF_F;
        }
}

// The same for groups of eight (or sixteen) query heads per KV head: a warp owns one position, the routing queries of
// eight heads are rows 0..7 of the A operand (rows 8..15 are zero), the columns of B are the keys of eight strides.
// Lane (r8, q) receives the scores of head r8 at strides s0 + 2q and s0 + 2q + 1, so that four lanes share a head; their
// sorted lists are merged two at a time.  Every key row is fetched once for eight heads.
// Bound by the latency of the key rows (a chunk half way through a long context reads them from DRAM) and by issue
// (four lists of K values per head).  4096 positions at 500001, 32/4 heads,
// K = 16: 1515 us with a warp per position and selection from shared memory (the kernel of the other group sizes),
// 484 us here, about 440 us with the tiles fetched a step ahead.
template <int K>
__global__ void __launch_bounds__(kWarps * 32, 2)
search_rows8(const bf16 *__restrict__ q_s, const bf16 *__restrict__ k, Call c, int32_t *__restrict__ out_anchor,
             float *__restrict__ out_score) {
    extern __shared__ float smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r8 = lane >> 2, q = lane & 3;
    // the tiles with the most strides (the last positions) start first
    const long long r = (long long)(gridDim.x - 1 - blockIdx.x) * kWarps + warp;
    if (r >= c.Lq) return;
    const int bg = blockIdx.y, g = bg % c.Hkv, b = bg / c.Hkv, h = g * c.G + blockIdx.z * 8 + r8;
    Words8 qa[2];
    chain_wait();
    {
        const bf16 *base = q_s + b * c.q_sb + (long long)h * c.q_sh + r * c.q_st + 16 * q;
        qa[0] = ldg256(base);
        qa[1] = ldg256(base + 64);
    }
    const int i = (int)(c.q_pos0 + r);   // positions fit 31 bits
    const int n = n_strides(c, i);
    // Algorithm 1: anchors inside the local window are no candidates; t_s lies in W iff offset(s) <= w
    const int s_min = c.window > 0 ? window_strides(c) : 0;
    const bf16 *kbase = k + b * c.kv_sb + g * c.kv_sh + 16 * q;
    const int kv_st = (int)c.kv_st;
    auto fetch = [&](int s0, Words8 (&kb)[2]) {   // column r8: the key of stride s0 + r8
        const int s = s0 + r8;
        int t = i + 1 - stride_offset(c, s < c.n_off || !c.off ? s : 0);
        if (s >= n) t = i;   // a valid row either way
        const bf16 *row = kbase + (long long)t * kv_st;
        kb[0] = ldg256(row);
        kb[1] = ldg256(row + 64);
    };
    RunningTop<K> top(smem + (size_t)warp * (2 * RunningTop<K>::CAP * 32), lane);
    // two independent accumulation chains, added at the end
    auto score = [&](const Words8 (&kb)[2], float &x0, float &x1) {
        float a0[4] = {0.f, 0.f, 0.f, 0.f}, a1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            mma_bf16_16816(a0, qa[0].w[2 * x], 0u, qa[0].w[2 * x + 1], 0u, kb[0].w[2 * x], kb[0].w[2 * x + 1]);
            mma_bf16_16816(a1, qa[1].w[2 * x], 0u, qa[1].w[2 * x + 1], 0u, kb[1].w[2 * x], kb[1].w[2 * x + 1]);
        }
        x0 = (a0[0] + a1[0]) * c.search_scale;
        x1 = (a0[1] + a1[1]) * c.search_scale;
    };
    // two B tiles of eight strides, each fetched again as soon as its scores are taken
    Words8 ka[2], kb[2];
    int s0 = s_min;
    float zero = 0.f;   // zero times the scores: NaN once one of them is not finite
    fetch(s0, ka);
    fetch(s0 + 8, kb);
    for (; s0 + 16 <= n; s0 += 16) {
        const int s = s0 + 2 * q;
        float xa, xb;
        score(ka, xa, xb);
        fetch(s0 + 16, ka);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s, xa, s + 1, xb);
        score(kb, xa, xb);
        fetch(s0 + 24, kb);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s + 8, xa, s + 9, xb);
    }
    if (s0 < n) {
        const int s = s0 + 2 * q;
        float xa, xb;
        score(ka, xa, xb);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s, s < n ? xa : -CUDART_INF_F, s + 1, s + 1 < n ? xb : -CUDART_INF_F);
        score(kb, xa, xb);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s + 8, s + 8 < n ? xa : -CUDART_INF_F, s + 9, s + 9 < n ? xb : -CUDART_INF_F);
    }

    const long long obase = (((long long)b * c.Hq + h) * c.Lq + r) * c.top_k;
    if (__any_sync(0xffffffffu, zero != 0.f)) {
        NextBest next;
#pragma unroll 1
        for (int j = 0; j < c.top_k; ++j) {
#pragma unroll 1
            for (int s1 = s_min; s1 < n; s1 += 8) {
                const int s = s1 + 2 * q;
                float xa, xb;
                fetch(s1, ka);
                score(ka, xa, xb);
                if (s < n) next.offer(s, xa);
                if (s + 1 < n) next.offer(s + 1, xb);
            }
            next.merge(1);
            next.merge(2);
            if (q == 0) {
                out_anchor[obase + j] = next.found() ? i + 1 - stride_offset(c, next.s) : -1;
                out_score[obase + j] = next.score();
            }
            next.take();
        }
        return;
    }
    float ex[K];
    int es[K];
    top.finish(ex, es);
    merge_pairs<K>(ex, es, 1);
    merge_pairs<K>(ex, es, 2);
#pragma unroll
    for (int j = 0; j < K; ++j)
        if ((j & 3) == q && j < c.top_k) {
            const bool on = es[j] != INT_MAX;
            out_anchor[obase + j] = on ? i + 1 - stride_offset(c, es[j]) : -1;
            out_score[obase + j] = on ? ex[j] : -CUDART_INF_F;
        }
}

template <int K>
cudaError_t launch_k(const bf16 *q_s, const bf16 *k, const Call &c, int32_t *oa, float *os, cudaStream_t st) {
    constexpr size_t smem = (size_t)kWarps * 2 * ListCap<K>::value * 32 * sizeof(float);
    const bool four = c.G == kG;
    void (*kern)(const bf16 *, const bf16 *, Call, int32_t *, float *) = four ? search_diag<K> : search_rows8<K>;
    static bool attr_set[64][2] = {};
    if (smem > 48 * 1024) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
        if (dev < 0 || dev >= 64 || !attr_set[dev][four]) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            if (dev >= 0 && dev < 64) attr_set[dev][four] = true;
        }
    }
    const int rows = kWarps * (four ? kQW : 1);   // positions per CTA
    const dim3 blocks((unsigned)((c.Lq + rows - 1) / rows), (unsigned)(c.B * c.Hkv), four ? 1u : (unsigned)(c.G / 8));
    return launch_chained(kern, blocks, dim3(kWarps * 32), smem, st, q_s, k, c, oa, os);
}

}  // namespace

bool search_diag_supported(const Call &c, int dtype) {
    // (the 32-byte loads want 32-byte aligned rows: strides in multiples of 16 elements)
    return dtype == SLA_BF16 && c.D == 128 && (c.G == kG || c.G % 8 == 0) && c.top_k <= 16 && (long long)c.B * c.Hkv <= 65535 &&
           c.kv_st <= INT_MAX && c.q_pos0 + c.Lq <= INT_MAX &&
           (c.q_sb | c.q_sh | c.q_st | c.kv_sb | c.kv_sh | c.kv_st) % 16 == 0;
}

cudaError_t launch_search_diag(const void *q_s, const void *k, const Call &c, int32_t *oa, float *os, cudaStream_t st,
                               long long *launches) {
    const bf16 *qs = (const bf16 *)q_s, *kk = (const bf16 *)k;
    cudaError_t e;
    if (c.top_k <= 2) e = launch_k<2>(qs, kk, c, oa, os, st);
    else if (c.top_k <= 4) e = launch_k<4>(qs, kk, c, oa, os, st);
    else if (c.top_k <= 8) e = launch_k<8>(qs, kk, c, oa, os, st);
    else e = launch_k<16>(qs, kk, c, oa, os, st);
    if (launches) *launches += 1;
    return e;
}

}  // namespace sla
