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
constexpr int kWarps = 4;
constexpr int kQW = 4;   // query positions per warp
constexpr int kG = 4;    // query heads per KV head

// Entries of a lane's list: of a hundred scores in random order 2 + 2 ln 50 = 10 are among the two best so far, 18, 28 and 45
// among the four, eight and sixteen best, and a list that runs full costs all lanes of the warp a pass over theirs.  (48 entries
// for K = 16 are what four CTAs of an SM have room for; with 52, which leave three, 4096 positions at 500001 took 496 us
// instead of 373.)
template <int K> struct ListCap { static constexpr int value = K == 2 ? 16 : K == 4 ? 24 : K == 8 ? 32 : 48; };

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The first of a chain: no accumulators to clear.
__device__ __forceinline__ void mma_bf16_16816_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                     uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
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

// A lane's running top-k: the K best values so far, sorted, in registers, and in shared memory (entry e at list[32 e]) every
// score with its stride index that beat the K-th best when it arrived.
template <int K>
struct RunningTop {
    static constexpr int CAP = ListCap<K>::value;
    float v[K];
    uint32_t list, end;   // shared-memory addresses of the lane's first entry and behind its last; 256 bytes from entry to entry
    __device__ __forceinline__ RunningTop(float2 *warp_lists, int lane)
        : list(static_cast<uint32_t>(__cvta_generic_to_shared(warp_lists + lane))), end(list) {
#pragma unroll
        for (int j = 0; j < K; ++j) v[j] = -CUDART_INF_F;
    }
    static __device__ __forceinline__ void put(uint32_t at, float x, int s) {
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(__float_as_int(x)), "r"(s) : "memory");
    }
    static __device__ __forceinline__ void get(uint32_t at, float &x, int &s) {
        int w;
        asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(w), "=r"(s) : "r"(at) : "memory");
        x = __int_as_float(w);
    }
    // Drops the list entries that can no longer be among the K best (all lanes, each its own list):
    // what is left are the entries above the K-th best value and the earliest of those equal to it,
    // at most K in all, still in stride order.
    __device__ __forceinline__ void compact() {
        const float vk = v[K - 1];
        int allow_eq = K;
#pragma unroll
        for (int j = 0; j < K; ++j) allow_eq -= v[j] > vk;
        uint32_t w = list;
        for (uint32_t e = list; e < end; e += 1024) {   // four loads at a time: the list is as long as a multiple of four
            float x[4];
            int s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) get(e + 256 * u, x[u], s[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool eq = x[u] == vk;
                if (e + 256 * u < end && (x[u] > vk || (eq && allow_eq > 0))) {
                    allow_eq -= eq;
                    put(w, x[u], s[u]);
                    w += 256;
                }
            }
        }
        end = w;
    }
    // Two new scores, sa < sb.  Each one that beats the K-th best so far goes to the list; the sorted values take
    // both in one pass: with hi >= lo the new j-th best is max(v[j], min(v[j-1], hi), min(v[j-2], lo)).
    __device__ __forceinline__ void offer2(int sa, float xa, int sb, float xb) {
        if (__any_sync(0xffffffffu, end - list >= 256 * (CAP - 1))) compact();   // room for both scores
        const float vk = v[K - 1];
        if (xa > vk) {
            put(end, xa, sa);
            end += 256;
        }
        if (xb > vk) {
            put(end, xb, sb);
            end += 256;
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
            get(list + 256 * j, x[j], s[j]);
            if (list + 256 * j >= end) {
                x[j] = -CUDART_INF_F;
                s[j] = INT_MAX;
            }
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

// What bounds search_diag: the latency of the key rows (L2, a step ahead of their use in 32 registers) and of the step's chains at
// 16 warps an SM; issue slots 48 % used, L2 at 45 %.  Operations taken out of the step -- accumulators cleared by moves, strides
// squared and compared per fetch, two stores and 64-bit addresses per list entry -- and CTAs of four warps instead of eight: 16384
// positions, 32/8 heads, K = 8 250 -> 227 us; 65536 1583 -> 1437; two sequences of 262144, 16/4 heads, K = 16 14.28 -> 12.46 ms;
// 32768, K = 2 751 -> 673 us.  Five CTAs an SM (96 registers) spill: 240 us for the first of these.
//
// The strides a lane fetches, one after another: key positions i + 1 - offset(s), i + 1 - offset(s + step), ...  On the
// quadratic pattern the distance to the next one, 2 step (s + 1) + step^2, itself grows by 2 step^2.  A position without the
// stride (s >= n) gets key 0: a valid row either way.
template <bool kTable>
struct KeyWalk {
    const char *base;
    unsigned pitch;       // bytes
    int t, d, s, dd;      // kTable: t the query position
    const int *off;
    int n;
    __device__ __forceinline__ KeyWalk(const bf16 *k, const Call &c, int i, int s0, int step, int n_)
        : base(reinterpret_cast<const char *>(k)), pitch((unsigned)c.kv_st * 2u), off(c.off), n(n_) {
        if constexpr (kTable) {
            t = i; s = s0; d = step;
        } else {
            t = s0 < n ? i + 1 - (s0 + 1) * (s0 + 1) : -1;   // (the square of a stride that exists fits 31 bits)
            d = step * (2 * (s0 + 1) + step);
            dd = 2 * step * step;
        }
    }
    __device__ __forceinline__ void next(Words8 (&kb)[2]) {
        unsigned at;
        if constexpr (kTable) {
            at = s < n ? (unsigned)(t + 1 - off[s]) : 0u;
            s += d;
        } else {
            at = (unsigned)max(t, 0);
            t -= d;
            d += dd;
        }
        const char *row = base + (unsigned long long)at * pitch;
        kb[0] = ldg256(row);
        kb[1] = ldg256(row + 128);
    }
};

template <int K, bool kTable>
__global__ void __launch_bounds__(kWarps * 32, 4)
search_diag(const bf16 *__restrict__ q_s, const bf16 *__restrict__ k, Call c, int32_t *__restrict__ out_anchor,
            float *__restrict__ out_score) {
    extern __shared__ float2 smem[];
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

    KeyWalk<kTable> walk(k + b * c.kv_sb + g * c.kv_sh + 16 * q, c, i_ld, s_min + u_ld, 2, n_ld);

    RunningTop<K> top(smem + (size_t)warp * (RunningTop<K>::CAP * 32), lane);
    // scores of one B tile (two strides): two independent accumulation chains, added at the end
    auto score = [&](const Words8 (&kb)[2]) -> float {
        float a0[4], a1[4];
        mma_bf16_16816_first(a0, qa[0].w[0], qb[0].w[0], qa[0].w[1], qb[0].w[1], kb[0].w[0], kb[0].w[1]);
        mma_bf16_16816_first(a1, qa[1].w[0], qb[1].w[0], qa[1].w[1], qb[1].w[1], kb[1].w[0], kb[1].w[1]);
#pragma unroll
        for (int x = 1; x < 4; ++x) {
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
    walk.next(ka);
    walk.next(kb);
    for (; s0 + 4 <= n_all; s0 += 4) {
        const float xa = score(ka);
        walk.next(ka);
        const float xb = score(kb);
        walk.next(kb);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s0 + u_own, xa, s0 + 2 + u_own, xb);
    }
    for (; s0 < n_max; s0 += 4) {
        const float xa = score(ka), xb = score(kb);
        const bool on_a = s0 + u_own < n_own, on_b = s0 + 2 + u_own < n_own;   // (key 0 stands in for the key of an absent stride)
        zero = fmaf(on_a ? xa : 0.f, 0.f, fmaf(on_b ? xb : 0.f, 0.f, zero));
        top.offer2(s0 + u_own, on_a ? xa : -CUDART_INF_F, s0 + 2 + u_own, on_b ? xb : -CUDART_INF_F);
        if (s0 + 4 < n_max) {
            walk.next(ka);
            walk.next(kb);
        }
    }

    const long long obase = ((((long long)b * c.Hq + g * kG + hh) * c.Lq) + r0 + jq) * c.top_k;
    if (__any_sync(0xffffffffu, zero != 0.f)) {
        NextBest next;
#pragma unroll 1
        for (int j = 0; j < c.top_k; ++j) {
#pragma unroll 1
            for (int s1 = s_min; s1 < n_max; s1 += 2) {
                KeyWalk<kTable>(k + b * c.kv_sb + g * c.kv_sh + 16 * q, c, i_ld, s1 + u_ld, 2, n_ld).next(ka);
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
// 484 us here, about 440 us with the tiles fetched a step ahead, 373 us (from 407 on the same GPU) with the shorter step.
// Half of the A operand is zero, so that five CTAs fit an SM up to K = 8 with few spills (24 bytes at K = 8, 44 with a table): 16384 positions, 32/4
// heads, K = 8 253 us with four CTAs, 234 with five; 2048 at 300000 141 and 120; K = 2 152 and 140, 123 and 102.
template <int K, bool kTable>
__global__ void __launch_bounds__(kWarps * 32, K <= 8 ? 5 : 4)
search_rows8(const bf16 *__restrict__ q_s, const bf16 *__restrict__ k, Call c, int32_t *__restrict__ out_anchor,
             float *__restrict__ out_score) {
    extern __shared__ float2 smem[];
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
    KeyWalk<kTable> walk(kbase, c, i, s_min + r8, 8, n);   // column r8: the keys of strides s_min + r8, + 8, ...
    RunningTop<K> top(smem + (size_t)warp * (RunningTop<K>::CAP * 32), lane);
    // two independent accumulation chains, added at the end
    auto score = [&](const Words8 (&kb)[2], float &x0, float &x1) {
        float a0[4], a1[4];
        mma_bf16_16816_first(a0, qa[0].w[0], 0u, qa[0].w[1], 0u, kb[0].w[0], kb[0].w[1]);
        mma_bf16_16816_first(a1, qa[1].w[0], 0u, qa[1].w[1], 0u, kb[1].w[0], kb[1].w[1]);
#pragma unroll
        for (int x = 1; x < 4; ++x) {
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
    walk.next(ka);
    walk.next(kb);
    for (; s0 + 16 <= n; s0 += 16) {
        const int s = s0 + 2 * q;
        float xa, xb;
        score(ka, xa, xb);
        walk.next(ka);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s, xa, s + 1, xb);
        score(kb, xa, xb);
        walk.next(kb);
        zero = fmaf(xa, 0.f, fmaf(xb, 0.f, zero));
        top.offer2(s + 8, xa, s + 9, xb);
    }
    if (s0 < n) {
        const int s = s0 + 2 * q;
        float xa, xb;
        auto offer_present = [&](int s) {   // (key 0 stands in for the key of an absent stride)
            zero = fmaf(s < n ? xa : 0.f, 0.f, fmaf(s + 1 < n ? xb : 0.f, 0.f, zero));
            top.offer2(s, s < n ? xa : -CUDART_INF_F, s + 1, s + 1 < n ? xb : -CUDART_INF_F);
        };
        score(ka, xa, xb);
        offer_present(s);
        score(kb, xa, xb);
        offer_present(s + 8);
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
                KeyWalk<kTable>(kbase, c, i, s1 + r8, 8, n).next(ka);
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
    const bool table = c.off != nullptr;
    void (*kern)(const bf16 *, const bf16 *, Call, int32_t *, float *) =
        four ? (table ? search_diag<K, true> : search_diag<K, false>) : table ? search_rows8<K, true> : search_rows8<K, false>;
    static_assert(smem <= 48 * 1024, "what a kernel without arrays of its own has without asking");
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
