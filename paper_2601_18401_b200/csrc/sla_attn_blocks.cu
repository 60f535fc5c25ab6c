// Span-attention of the generic layouts (fp32, head_dim 64, broadcast K/V) by blocks of keys, union mode.
//
// With one warp per query row every selected key row travels from L2 to an SM once per query row; at 4096 positions,
// top_k 4 and spans of 129 keys that is 1 GB, or 52 us at the L2's rate for two megabytes of keys and values.  Here a CTA
// keeps 64 keys and values in shared memory and serves every query row of its share that selected any of them:
//   scan    each thread reads the anchors of a row and forms the 64-bit mask of the block's keys that lie in the row's
//           spans (the union is the OR of the spans' masks: no sorting, no clipping); rows with a mask go to a list;
//   attend  a warp takes LPR lanes x up to 4 rows per group (32 rows at head_dim 64, 16 at 128): a lane holds 16 dims of four
//           query rows, reads the same 16 dims of a key as its group's peers (broadcast) and the lanes' sums are exchanged
//           so that each lane ends up with the score of one row; the 64 keys, then the exponentials, then the values
//           (every row multiplies all 64, with weight 0 where it did not select the key: an Inf or NaN among them is
//           zero in shared memory and comes from global memory for the rows that did);
//   merge   a row has one partial result per key block it touches, at a slot that only the row's own spans determine
//           (first span that reaches the block, block within that span), combined in slot order.
// Everything is fp32 FMA (two per instruction), as in the row kernel: bf16 inputs are widened exactly.
// Bound by the FMA pipe and, at 12 to 16 warps an SM, by the latency of its chains: 64 f32x2 products per key and 32 rows
// (issue slots 40 % used; two thirds of the products belong to selected keys).  Search and attention together,
// row kernel and this one: 4096 positions, one head of 64 dims, top_k 4, spans of 129 keys 88 and 52 us; 3811 positions, one
// head of 128 dims, top_k 8, spans of up to 125 keys 258 and 100 us; 7343 positions, two heads, 173 keys 479 and 301 us.
#include <limits.h>
#include <math_constants.h>

#include <type_traits>

#include "sla_kernels.h"

namespace sla {

namespace {

constexpr int kKeys = 64;        // keys of a block
constexpr int kPitch = kKeys + 4;
constexpr int kList = 512;       // rows a CTA collects before it attends
constexpr int kMergeWarps = 4;
constexpr size_t kScratchTarget = 80u << 20;   // partial results of a chunk of rows: they stay in L2

template <int D> struct Tile {
    static constexpr int LPR = D / 16;        // lanes per group of four rows
    static constexpr int NG = 32 / LPR;       // groups per warp
    static constexpr int ROWS = 4 * NG;
    static constexpr int WARPS = D == 64 ? 4 : 8, CTAS = D == 64 ? 3 : 2;   // 12 or 16 warps on an SM
    static constexpr size_t smem = sizeof(float) * (2 * kKeys * D + WARPS * ROWS * kPitch) + sizeof(int4) * kList + 16;
};

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

// Keys of block kb in [lo, hi] as a mask.
__device__ __forceinline__ unsigned long long span_mask(int lo, int hi, int k0) {
    const int a = lo - k0 > 0 ? lo - k0 : 0, z = hi - k0 < kKeys - 1 ? hi - k0 : kKeys - 1;
    return a <= z ? (~0ull >> (kKeys - 1 - z)) & (~0ull << a) : 0ull;
}

struct BlockPlan {
    int span_blocks, window_blocks, slots;   // key blocks a span, the window, a row can touch
    int Lc;                                  // rows of a chunk
    size_t o_ml, o_part, bytes;
    Canaries canaries;
};

// One row's interval j: span of anchor j, or the window for j == top_k; empty (hi < lo) if there is none.
__device__ __forceinline__ void interval(const Call &c, int t, int j, int i, long long ell, int &lo, int &hi) {
    lo = INT_MAX;
    hi = -1;
    if (j == c.top_k && c.window > 0) {
        lo = i - c.window + 1 > 0 ? i - c.window + 1 : 0;
        hi = i;
        return;
    }
    if (t < 0 || t > i) return;
    const long long a = t - (long long)c.back * ell, z = t + (long long)c.fwd * ell;
    lo = (int)(a > 0 ? a : 0);
    hi = (int)(z < i ? z : i);
}

template <typename T, int D>
__global__ void __launch_bounds__(Tile<D>::WARPS * 32, Tile<D>::CTAS)
attend_blocks(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, Call c, BlockPlan p, int r_first,
              int n_rows, int share, const int32_t *__restrict__ anchor, float2 *__restrict__ ml, float *__restrict__ part) {
    using TL = Tile<D>;
    constexpr int LPR = TL::LPR, NG = TL::NG, ROWS = TL::ROWS, kWarps = TL::WARPS, kThreads = kWarps * 32;
    constexpr int E = Vec16<T>::kElems;
    extern __shared__ float4 smem4[];
    float *ks = reinterpret_cast<float *>(smem4), *vs = ks + kKeys * D, *ps = vs + kKeys * D;
    int4 *list = reinterpret_cast<int4 *>(ps + kWarps * ROWS * kPitch);   // row in the chunk, slot, mask
    int *count = reinterpret_cast<int *>(list + kList);
    unsigned *odd = reinterpret_cast<unsigned *>(count + 1);               // two words: keys whose values are not all finite
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = blockIdx.x * kKeys;
    const int g = blockIdx.y % c.Hkv, b = blockIdx.y / c.Hkv;
    // the rows at or after the block's first key, heads of the group one after another, in chunks of 32 dealt out in turn to
    // the block's CTAs (rows close after the block select it far more often than later ones: with contiguous shares 83 us
    // instead of 69 us, search included, at 2379 positions, two heads of 128 dims, K = 2)
    const long long before = k0 - (c.q_pos0 + r_first);
    const int r_lo = before > 0 ? (int)before : 0, nr = n_rows - r_lo;
    const int y_end = nr * c.G, n_ctas = (y_end + share - 1) / share;
    if ((int)blockIdx.z >= n_ctas) return;
    const int n_keys = (int)(c.q_pos0 + r_first + n_rows - k0 < kKeys ? c.q_pos0 + r_first + n_rows - k0 : kKeys);

    chain_wait();
    chain_release();
    const T *kbase = k + b * c.kv_sb + g * c.kv_sh + (long long)k0 * c.kv_st;
    const T *vbase = v + b * c.kv_sb + g * c.kv_sh + (long long)k0 * c.kv_st;
    for (int x = threadIdx.x; x < kKeys * (D / E); x += kThreads) {
        const int j = x / (D / E), d = x % (D / E) * E;
        if constexpr (sizeof(T) == 4) {   // lands while the anchors are scanned; rows past the last key are zero
            const long long src = (long long)(j < n_keys ? j : 0) * c.kv_st + d;
            const int bytes = j < n_keys ? 16 : 0;
            const uint32_t kd = (uint32_t)__cvta_generic_to_shared(ks + j * D + d), vd = (uint32_t)__cvta_generic_to_shared(vs + j * D + d);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(kd), "l"(kbase + src), "r"(bytes) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(vd), "l"(vbase + src), "r"(bytes) : "memory");
            continue;
        }
        float kf[E] = {}, vf[E] = {};
        if (j < n_keys) {
            Vec16<T>::load(kbase + j * c.kv_st + d, kf);
            Vec16<T>::load(vbase + j * c.kv_st + d, vf);
        }
#pragma unroll
        for (int e = 0; e < E; e += 4) {
            *reinterpret_cast<float4 *>(ks + j * D + d + e) = make_float4(kf[e], kf[e + 1], kf[e + 2], kf[e + 3]);
            *reinterpret_cast<float4 *>(vs + j * D + d + e) = make_float4(vf[e], vf[e + 1], vf[e + 2], vf[e + 3]);
        }
    }
    if (threadIdx.x == 0) *count = odd[0] = odd[1] = 0;
    __syncthreads();

    const int sub = lane / NG, grp = lane % NG;
    const float scale2 = c.softmax_scale * kLog2e;
    float *pw = ps + warp * ROWS * kPitch;
    const float *kl = ks + sub * 4, *vl = vs + sub * 4;

    // one pass of the warp over the block: R rows per group, entries e0 + r NG + grp of the list
    auto pass = [&](auto rows_per_group, int e0, int n) {
        constexpr int R = decltype(rows_per_group)::value;
        // the lane's own row (the one whose scores it receives): row sub & 3 of its group
        const int own = (sub & 3) < R ? e0 + (sub & 3) * NG + grp : n;
        int4 mine = make_int4(0, 0, 0, 0);
        if (own < n) mine = list[own];
        const T *qrow[R];
        float2 qv[R][8];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = e0 + r * NG + grp;
            const int row = list[e < n ? e : n - 1].x, rc = row % n_rows, hg = row / n_rows;
            qrow[r] = q + b * c.q_sb + (long long)(g * c.G + hg) * c.q_sh + (long long)(r_first + rc) * c.q_st + sub * 4;
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                float f[4];
                if constexpr (sizeof(T) == 4) {
                    const float4 w = __ldg(reinterpret_cast<const float4 *>(qrow[r] + x * 4 * LPR));
                    f[0] = w.x; f[1] = w.y; f[2] = w.z; f[3] = w.w;
                } else {
                    const uint2 w = __ldg(reinterpret_cast<const uint2 *>(qrow[r] + x * 4 * LPR));
                    f[0] = __uint_as_float(w.x << 16); f[1] = __uint_as_float(w.x & 0xffff0000u);
                    f[2] = __uint_as_float(w.y << 16); f[3] = __uint_as_float(w.y & 0xffff0000u);
                }
                qv[r][2 * x] = make_float2(f[0] * scale2, f[1] * scale2);
                qv[r][2 * x + 1] = make_float2(f[2] * scale2, f[3] * scale2);
            }
        // scores of the 64 keys, masked, to shared memory
        float m = -CUDART_INF_F, l = 0.f;
#pragma unroll 1
        for (int j = 0; j < kKeys; j += 4) {
            const unsigned mask = (j < 32 ? (unsigned)mine.z : (unsigned)mine.w) >> (j & 31);
            float s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float2 t[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) t[r] = make_float2(0.f, 0.f);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float4 w = *reinterpret_cast<const float4 *>(kl + (j + u) * D + x * 4 * LPR);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        t[r] = fma2(qv[r][2 * x], make_float2(w.x, w.y), t[r]);
                        t[r] = fma2(qv[r][2 * x + 1], make_float2(w.z, w.w), t[r]);
                    }
                }
                const float t0 = t[0].x + t[0].y, t1 = t[1].x + t[1].y, t2 = t[2].x + t[2].y, t3 = t[3].x + t[3].y;
                const float ya = ((sub & 1) ? t1 : t0) + __shfl_xor_sync(0xffffffffu, (sub & 1) ? t0 : t1, NG);
                const float yb = ((sub & 1) ? t3 : t2) + __shfl_xor_sync(0xffffffffu, (sub & 1) ? t2 : t3, NG);
                float z = ((sub & 2) ? yb : ya) + __shfl_xor_sync(0xffffffffu, (sub & 2) ? ya : yb, 2 * NG);
                if (LPR == 8) z += __shfl_xor_sync(0xffffffffu, z, 4 * NG);
                s[u] = (mask >> u) & 1u ? z : -CUDART_INF_F;
                m = fmaxf(m, s[u]);
            }
            if (sub < 4) *reinterpret_cast<float4 *>(pw + lane * kPitch + j) = make_float4(s[0], s[1], s[2], s[3]);
        }
        // exponentials of the lane's own row
        const float ref = m == -CUDART_INF_F ? 0.f : m;
        if (sub < 4) {
#pragma unroll 2
            for (int j = 0; j < kKeys; j += 4) {
                float4 *w = reinterpret_cast<float4 *>(pw + lane * kPitch + j);
                float4 x = *w;
                x.x = exp2f(x.x - ref); x.y = exp2f(x.y - ref); x.z = exp2f(x.z - ref); x.w = exp2f(x.w - ref);
                l += (x.x + x.y) + (x.z + x.w);
                *w = x;
            }
        }
        __syncwarp();
        // values
        float2 acc[R][8];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int x = 0; x < 8; ++x) acc[r][x] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int j = 0; j < kKeys; j += 4) {
            float pr[R][4];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 w = *reinterpret_cast<const float4 *>(pw + (r * NG + grp) * kPitch + j);
                pr[r][0] = w.x; pr[r][1] = w.y; pr[r][2] = w.z; pr[r][3] = w.w;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float4 w = *reinterpret_cast<const float4 *>(vl + (j + u) * D + x * 4 * LPR);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float2 pp = make_float2(pr[r][u], pr[r][u]);
                        acc[r][2 * x] = fma2(pp, make_float2(w.x, w.y), acc[r][2 * x]);
                        acc[r][2 * x + 1] = fma2(pp, make_float2(w.z, w.w), acc[r][2 * x + 1]);
                    }
                }
        }
        for (unsigned long long keys = odd[0] | (unsigned long long)odd[1] << 32; keys; keys &= keys - 1) {
            const int j = __ffsll((long long)keys) - 1;
            const T *row = vbase + (long long)j * c.kv_st + sub * 4;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int e = e0 + r * NG + grp;
                if (e >= n || !(((j < 32 ? (unsigned)list[e].z : (unsigned)list[e].w) >> (j & 31)) & 1u)) continue;
                const float w = pw[(r * NG + grp) * kPitch + j];
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    const T *at = row + (x >> 1) * 4 * LPR + (x & 1) * 2;
                    const float a = (float)at[0], z = (float)at[1];
                    if (!isfinite(a)) acc[r][x].x = fmaf(w, a, acc[r][x].x);
                    if (!isfinite(z)) acc[r][x].y = fmaf(w, z, acc[r][x].y);
                }
            }
        }
        __syncwarp();   // the next scores go to the same place
        if (own < n && sub < 4) ml[mine.y] = make_float2(m, l);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = e0 + r * NG + grp;
            if (e < n) {
                float *o = part + (size_t)list[e].y * D + sub * 4;
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    *reinterpret_cast<float4 *>(o + x * 4 * LPR) =
                        make_float4(acc[r][2 * x].x, acc[r][2 * x].y, acc[r][2 * x + 1].x, acc[r][2 * x + 1].y);
            }
        }
    };
    // The list in as few passes as four rows per group allow, its rows shared out evenly among the warps, the passes nearly equal:
    // a list of 92 rows is three rows per group in all four warps instead of four in three of them, one of 136 rows two passes of
    // three and two.  Search and attention: 4096 positions, one head, four spans 56.5 and 52.6 us; 8000, four heads 452 and 422; bf16,
    // 8192, four heads 428 and 388.  (At head_dim 128 the registers do not suffice: 3811 positions, eight spans 101 and 104 us.)
    auto attend = [&](int n) {
        if constexpr (D == 128) {
            for (int e0 = warp * ROWS; e0 < n; e0 += kWarps * ROWS) pass(std::integral_constant<int, 4>(), e0, n);
        } else {
            int units = (n + kWarps * NG - 1) / (kWarps * NG);   // rows per group still to come
            for (int passes = (units + 3) / 4, e0 = 0; passes > 0; --passes) {
                const int rows = (units + passes - 1) / passes, at = e0 + warp * NG * rows;
                if (at < n) {
                    if (rows == 4) pass(std::integral_constant<int, 4>(), at, n);
                    else if (rows == 3) pass(std::integral_constant<int, 3>(), at, n);
                    else if (rows == 2) pass(std::integral_constant<int, 2>(), at, n);
                    else pass(std::integral_constant<int, 1>(), at, n);
                }
                units -= rows;
                e0 += kWarps * NG * rows;
            }
        }
    };

    const int n_iv = c.top_k + (c.window > 0 ? 1 : 0);
    const int chunks = (y_end + 31) / 32;
    int ch = blockIdx.z + warp * n_ctas;   // the warp's next chunk
    bool more, staged = false;
    do {
        // as many chunks as the list has room for, without a barrier between them
        for (int it = 0; it < kList / kThreads && ch < chunks; ++it, ch += kWarps * n_ctas) {
            const int y = ch * 32 + lane, hg = y / nr, rc = r_lo + (y - hg * nr);
            unsigned long long mask = 0;
            int slot = 0;
            const long long row_all = ((long long)b * c.Hq + g * c.G + hg);
            if (y < y_end) {
                const int i = (int)(c.q_pos0 + r_first + rc);
                const long long ell = base_len(c, i);
                const int32_t *a = anchor + (row_all * c.Lq + r_first + rc) * c.top_k;
                for (int j0 = 0; j0 < n_iv; j0 += 4) {
                    int t[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) t[x] = j0 + x < c.top_k ? __ldg(a + j0 + x) : -1;
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        int lo, hi;
                        interval(c, t[x], j0 + x, i, ell, lo, hi);
                        const unsigned long long mj = span_mask(lo, hi, k0);
                        if (mj && !mask) slot = (j0 + x) * p.span_blocks + ((int)blockIdx.x - lo / kKeys);
                        mask |= mj;
                    }
                }
            }
            const unsigned on = __ballot_sync(0xffffffffu, mask != 0);
            int base = 0;
            if (lane == 0 && on) base = atomicAdd(count, __popc(on));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (mask)
                list[base + __popc(on & ((1u << lane) - 1u))] =
                    make_int4(hg * n_rows + rc, (int)((row_all * n_rows + rc) * p.slots + slot), (int)(unsigned)mask, (int)(unsigned)(mask >> 32));
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (!staged) {   // the values this thread brought in: zero times their sum is zero if all are finite
            staged = true;
            float4 *mine = reinterpret_cast<float4 *>(vs) + threadIdx.x;
            constexpr int kMine = kKeys * D / 4 / kThreads;
            float zero = 0.f;
#pragma unroll
            for (int u = 0; u < kMine; ++u) {
                const float4 w = mine[u * kThreads];
                zero += w.x * 0.f + w.y * 0.f + (w.z * 0.f + w.w * 0.f);
            }
            if (zero != 0.f)
#pragma unroll 1
                for (int u = 0; u < kMine; ++u) {
                    const float4 w = mine[u * kThreads];
                    if (isfinite(w.x) && isfinite(w.y) && isfinite(w.z) && isfinite(w.w)) continue;
                    mine[u * kThreads] = make_float4(isfinite(w.x) ? w.x : 0.f, isfinite(w.y) ? w.y : 0.f, isfinite(w.z) ? w.z : 0.f,
                                                     isfinite(w.w) ? w.w : 0.f);
                    const int j = (threadIdx.x + u * kThreads) / (D / 4);
                    atomicOr(odd + j / 32, 1u << (j % 32));
                }
        }
        more = __syncthreads_or(ch < chunks);
        attend(*count);
        if (more) {
            __syncthreads();
            if (threadIdx.x == 0) *count = 0;
            __syncthreads();
        }
    } while (more);
}

// One warp per row: the partial results of the blocks its spans touch, in slot order.
template <typename T, int D>
__global__ void __launch_bounds__(kMergeWarps * 32)
merge_blocks(Call c, BlockPlan p, int r_first, int n_rows, const int32_t *__restrict__ anchor, const float2 *__restrict__ ml,
             const float *__restrict__ part, T *__restrict__ out, float *__restrict__ lse) {
    constexpr int LPR = D / 4, NP = 32 / LPR;   // lanes per partial result, partial results per load
    constexpr int kIv = kMaxTopK + 1;
    __shared__ int s_b0[kMergeWarps][kIv], s_b1[kMergeWarps][kIv];
    __shared__ int s_at[kMergeWarps][32];
    __shared__ float s_w[kMergeWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long row = (long long)blockIdx.x * kMergeWarps + warp;   // (b, h, row of the chunk)
    if (row >= (long long)c.B * c.Hq * n_rows) return;
    const long long bh = row / n_rows;
    const int rc = (int)(row - bh * n_rows), h = (int)(bh % c.Hq), b = (int)(bh / c.Hq);
    const int i = (int)(c.q_pos0 + r_first + rc);
    const long long ell = base_len(c, i), orow = bh * c.Lq + r_first + rc;
    const int n_iv = c.top_k + (c.window > 0 ? 1 : 0);
    const int32_t *a = anchor + orow * c.top_k;
    for (int j = lane; j < n_iv; j += 32) {
        int lo, hi;
        const int t = j < c.top_k ? __ldg(a + j) : -1;
        interval(c, t, j, i, ell, lo, hi);
        if (t > i) atomicOr(c.status, kStatusBadIndex);
        s_b0[warp][j] = lo / kKeys;
        s_b1[warp][j] = hi < 0 ? -1 : hi / kKeys;
    }
    __syncwarp();
    chain_wait();
    const int sub = lane % LPR, half = lane / LPR;
    float M = -CUDART_INF_F, L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < p.slots; c0 += 32) {
        const int s = c0 + lane;
        bool valid = s < p.slots;
        float2 w = make_float2(-CUDART_INF_F, 0.f);
        if (valid) {
            const int j = s / p.span_blocks < c.top_k ? s / p.span_blocks : c.top_k;
            const int x = s_b0[warp][j] + (s - j * p.span_blocks);
            valid = x <= s_b1[warp][j];
            for (int y = 0; y < j; ++y) valid = valid && !(s_b0[warp][y] <= x && x <= s_b1[warp][y]);
            if (valid) w = ml[row * p.slots + s];
        }
        const unsigned on = __ballot_sync(0xffffffffu, valid);
        if (!on) continue;
        float mx = w.x;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float mn = fmaxf(M, mx), corr = exp2f(M - mn), f = valid ? exp2f(w.x - mn) : 0.f;
        float sum = w.y * f;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        L = L * corr + sum;
        M = mn;
        acc.x *= corr; acc.y *= corr; acc.z *= corr; acc.w *= corr;
        __syncwarp();
        if (valid) {
            const int at = __popc(on & ((1u << lane) - 1u));
            s_at[warp][at] = s;
            s_w[warp][at] = f;
        }
        __syncwarp();
        const int n = __popc(on);
#pragma unroll 4
        for (int x = half; x < n; x += NP) {
            const float4 o = __ldg(reinterpret_cast<const float4 *>(part + (size_t)(row * p.slots + s_at[warp][x]) * D) + sub);
            const float wx = s_w[warp][x];
            acc.x = fmaf(wx, o.x, acc.x); acc.y = fmaf(wx, o.y, acc.y); acc.z = fmaf(wx, o.z, acc.z); acc.w = fmaf(wx, o.w, acc.w);
        }
    }
    if (NP == 2) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 16);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 16);
        acc.z += __shfl_xor_sync(0xffffffffu, acc.z, 16);
        acc.w += __shfl_xor_sync(0xffffffffu, acc.w, 16);
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
    if (half == 0) {
        T *o = out + b * c.q_sb + (long long)h * c.q_sh + (long long)(r_first + rc) * c.q_st + sub * 4;
        o[0] = from_float<T>(acc.x * inv); o[1] = from_float<T>(acc.y * inv);
        o[2] = from_float<T>(acc.z * inv); o[3] = from_float<T>(acc.w * inv);
    }
    if (lane == 0) lse[orow] = L > 0.f ? (M + log2f(L)) * kLn2 : -CUDART_INF_F;
}

template <typename T, int D>
cudaError_t launch_t(const T *q, const T *k, const T *v, const Call &c, const BlockPlan &p, int r0, int n, const int32_t *anchor,
                     char *ws, T *out, float *lse, int sm_count, cudaStream_t st) {
    constexpr size_t smem = Tile<D>::smem;
    auto kern = attend_blocks<T, D>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    float2 *ml = reinterpret_cast<float2 *>(ws + p.o_ml);
    float *part = reinterpret_cast<float *>(ws + p.o_part);
    const long long blocks = (c.q_pos0 + r0 + n + kKeys - 1) / kKeys, bg = (long long)c.B * c.Hkv;
    // Shares of equal numbers of rows: as many CTAs as the chip holds at a time, or a multiple of that where the blocks
    // are many.  Every block's last share is a part of one: 0.6 of a CTA per block is set aside for them, so that no
    // few CTAs are left for a wave of their own (rounded up to the next chunk of rows alone: 10 % more at 7343 rows).
    const long long full = (c.q_pos0 + r0) / kKeys + 1 < blocks ? (c.q_pos0 + r0) / kKeys + 1 : blocks;   // blocks that every row may select
    long long scanned = full * n;
    for (long long x = full; x < blocks; ++x) scanned += n - (x * kKeys - (c.q_pos0 + r0));
    const long long chip = (long long)Tile<D>::CTAS * sm_count, waves = (2 * blocks * bg + chip - 1) / chip;
    const long long ctas = waves * chip - blocks * bg * 6 / 10;
    const int share = (int)(((scanned * bg * c.G + ctas - 1) / ctas + 31) / 32 * 32);
    const long long z = ((long long)n * c.G + share - 1) / share;
    cudaError_t e = launch_chained(kern, dim3((unsigned)blocks, (unsigned)bg, (unsigned)z), dim3(Tile<D>::WARPS * 32), smem, st, q, k, v, c, p,
                                   r0, n, share, anchor, ml, part);
    if (e != cudaSuccess) return e;
    const long long rows = (long long)c.B * c.Hq * n;
    return launch_chained(merge_blocks<T, D>, dim3((unsigned)((rows + kMergeWarps - 1) / kMergeWarps)), dim3(kMergeWarps * 32), 0, st, c, p, r0,
                          n, anchor, (const float2 *)ml, (const float *)part, out, lse);
}

// Scratch for chunks of at most `rows` query positions; ok = false where the kernel does not apply.
bool plan(const Call &c, long long rows, size_t gap, BlockPlan &p) {
    const long long i_last = c.q_pos0 + c.Lq - 1;
    const long long len = (long long)(c.back + c.fwd) * base_len(c, i_last) + 1;
    const long long sb = (len + kKeys - 2) / kKeys + 1, wb = c.window > 0 ? (c.window + kKeys - 2) / kKeys + 1 : 0;
    const long long slots = c.top_k * sb + wb, bh = (long long)c.B * c.Hq;
    if (slots > 65536 || rows < 1 || bh * rows * slots > INT_MAX) return false;
    p.span_blocks = (int)sb;
    p.window_blocks = (int)wb;
    p.slots = (int)slots;
    p.Lc = (int)rows;
    p.canaries = Canaries();
    size_t off = 0;
    auto region = [&](size_t size) {
        if (gap) { p.canaries.add(off); off += gap; }
        const size_t at = off;
        off += (size + 255) / 256 * 256;
        return at;
    };
    p.o_ml = region(sizeof(float2) * bh * rows * slots);
    p.o_part = region(sizeof(float) * c.D * bh * rows * slots);
    if (gap) { p.canaries.add(off); off += gap; }
    p.bytes = off;
    return true;
}

// Rows of a chunk whose partial results take at most `bytes` (0: not even one).
long long rows_for(const Call &c, size_t bytes, size_t gap) {
    BlockPlan one;
    if (!plan(c, 1, gap, one)) return 0;
    const size_t per_row = (sizeof(float2) + sizeof(float) * c.D) * (size_t)c.B * c.Hq * one.slots;
    const size_t fixed = 3 * gap + 512;
    long long rows = bytes > fixed ? (long long)((bytes - fixed) / per_row) : 0;
    if (rows > c.Lq) rows = c.Lq;
    return rows;
}

// Rows of the chunks the kernel is given the scratch for.
long long target_rows(const Call &c, size_t gap) {
    return rows_for(c, kScratchTarget, gap);
}

}  // namespace

// Which of the two kernels, from what each of them does (microseconds; the factors are fitted to 898 calls of both kernels
// over rows 1..8000, positions up to 400000, 1..64 spans of 2..3700 keys, and are off by 15 % in the median; the calls were timed
// before a list's rows were shared out evenly among the warps, which took 7 to 10 % off the blocks at head_dim 64):
//   by rows    a warp's walk over its row, one step per span and per two loads of a warp (a row or more of keys each); the
//              pieces it sorts; the products of selected keys
//   by blocks  per chunk of rows a launch of two kernels and 64 staged keys and values per CTA, whether any row selects
//              them or not; the anchors that every CTA scans; the products of whole blocks of selected keys; the slots a
//              row's merge looks through
// The blocks have to be a fifth better, which keeps calls with the row kernel where the two estimates lie close.  Over 500
// other calls that is 2 % above the better kernel in the mean, and 1 call more than 5 % slower than by rows (a rule by the
// number of rows and slots before it: 105 calls, up to 50 times).  The attention alone by rows and by blocks: 500 x 2 rows at
// 200000, 128 dims, four spans of 895 keys 1707 and 580 us; 16 x 8 rows at 1000000, four spans of 65 keys 55 and 1110 us;
// 1 x 8 rows at 300000, 64 dims, the same spans 32 and 180 us; 256 x 4 rows at 60000, two spans of 129 keys 28 and 147 us.
static bool blocks_are_faster(const Call &c, int dtype, const BlockPlan &p) {
    const long long i_last = c.q_pos0 + c.Lq - 1, len = (long long)(c.back + c.fwd) * base_len(c, i_last) + 1;
    const double rows = (double)c.B * c.Hq * c.Lq, blocks = (double)(i_last / kKeys + 1), bg = (double)c.B * c.Hkv;
    const double strides = n_strides(c, i_last), spans = c.top_k < strides ? c.top_k : strides;
    const double wanted = (double)c.top_k * len + c.window, keys = wanted < i_last + 1 ? wanted : i_last + 1;
    const double per_load = 32.0 / (c.D * (dtype == SLA_F32 ? 4 : 2) / 16);   // keys a load of a warp covers
    const double by_rows = 9 + 0.30 * (spans + keys / (2 * per_load)) + 0.26e-4 * rows * c.top_k + 26e-8 * rows * keys * c.D;
    const double near = spans * ((len - 1) / (double)kKeys + 1) + (c.window > 0 ? c.window / (double)kKeys + 1 : 0);
    const double touched = near < blocks ? near : blocks, chunks = (double)((c.Lq + p.Lc - 1) / p.Lc);
    const double by_blocks = chunks * (16 + 13e-5 * blocks * bg * c.D) +
                             7.5e-6 * blocks * bg * c.Lq * c.G * (c.top_k + (c.window > 0 ? 1 : 0)) +
                             5.3e-6 * rows * touched * c.D + 1.5e-3 * p.slots * c.top_k;
    return by_blocks < 0.8 * by_rows;
}

bool attn_blocks_supported(const Call &c, int dtype) {
    if (c.mode != SLA_UNION || (c.D != 64 && c.D != 128) || (long long)c.B * c.Hkv > 65535) return false;
    BlockPlan p;
    const long long rows = target_rows(c, 0);
    return rows >= 1 && plan(c, rows, 0, p) && blocks_are_faster(c, dtype, p);
}

size_t attn_blocks_bytes(const Call &c, size_t gap) {
    BlockPlan p;
    return plan(c, target_rows(c, gap), gap, p) ? p.bytes : 0;
}

// Rows per chunk in `avail` bytes of scratch; 0 if that is not half of what attn_blocks_bytes gives room for.
long long attn_blocks_rows(const Call &c, size_t avail, size_t gap) {
    const long long rows = rows_for(c, avail < kScratchTarget ? avail : kScratchTarget, gap);
    return 2 * rows >= target_rows(c, gap) ? rows : 0;
}

cudaError_t launch_attn_blocks(const void *q, const void *k, const void *v, const Call &c, int dtype, const int32_t *anchor,
                               long long step, void *out, float *lse, char *ws, int sm_count, bool canaries, cudaStream_t st, long long *launches) {
    const size_t gap = canaries ? Canaries::kBytes : 0;
    BlockPlan p;
    if (!plan(c, step, gap, p)) return cudaErrorInvalidValue;
    for (long long r0 = 0; r0 < c.Lq; r0 += step) {
        const int n = (int)(c.Lq - r0 < step ? c.Lq - r0 : step);
        cudaError_t e = cudaSuccess;
        if (canaries) e = launch_canary_fill(ws, p.canaries, st);
        if (e != cudaSuccess) return e;
#define SLA_BLOCKS(T, D) launch_t<T, D>((const T *)q, (const T *)k, (const T *)v, c, p, (int)r0, n, anchor, ws, (T *)out, lse, sm_count, st)
        if (dtype == SLA_F32) e = c.D == 64 ? SLA_BLOCKS(float, 64) : SLA_BLOCKS(float, 128);
        else e = c.D == 64 ? SLA_BLOCKS(__nv_bfloat16, 64) : SLA_BLOCKS(__nv_bfloat16, 128);
#undef SLA_BLOCKS
        if (e == cudaSuccess && canaries) e = launch_canary_check(ws, p.canaries, c.status, st);
        if (e != cudaSuccess) return e;
        *launches += 2;
    }
    return cudaSuccess;
}

}  // namespace sla
