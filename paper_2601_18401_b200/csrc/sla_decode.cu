// Decode step of libsla (Section "Kernel design", paragraph "Decoding path"): routing scores over
// the anchors of the single query position i = n_ctx-1, top-k, then attention over the routed spans
// read from the KV cache.  The step is bound by HBM reads of the selected K/V rows, so the attention
// kernel spreads each head's tokens evenly over many CTAs (split-K), streams whole rows with 16-byte
// loads, keeps a running (max, denominator, numerator) per lane group and merges at the end.
//
//   decode_attn    grid (CTAs per attention unit, units).  Where the anchors of a head fit a cluster of up to 8 CTAs it is
//                  the whole step in one launch: each CTA of the cluster scores a share of the anchors and writes the scores to
//                  all of them (distributed shared memory); otherwise the scores come from decode_score, launched before
//                  it (plan_decode).  Every CTA then selects the k best of its head itself, builds the spans of its
//                  unit, clips the overlaps and runs the online softmax over an even share of the tokens; the
//                  cluster's first CTA merges its partial results through their log-sum-exp, the last cluster of a unit
//                  those of the clusters.
//                  Union mode: one unit per head (its spans and the local window, clipped to disjoint pieces).
//                  Per-span mode (Algorithm 1 literally): one unit per selected anchor, J_t = S_t united with
//                  the window; the unit that finishes a head last applies the gate of Section "Combination" to
//                  the units' outputs.
//   decode_score   grid (anchor chunks, B*Hkv, head tiles): K anchor rows x G routing queries -> scores.  In the
//                  sequence-sharded step the CTA that finishes a (batch, KV head) last selects this rank's k best candidates.
// "Last" is decided by an atomic counter per unit / per head in the handle's header region; the last CTA puts
// the counter back to zero, so a step leaves them as it found them.
#include <cooperative_groups.h>
#include <limits.h>
#include <math_constants.h>

#include "sla_kernels.h"
#include "sla_topk.cuh"

namespace sla {

namespace cg = cooperative_groups;

namespace {

constexpr int kScoreThreads = 256;
constexpr int kAttnThreads = 256;

template <int LPR> __device__ inline float reduce_sub(float x) {
#pragma unroll
    for (int off = LPR / 2; off >= 1; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}

// ------------------------------------------------------------------------------------------------
template <typename T, int D, int GT>
__global__ void __launch_bounds__(kScoreThreads)
decode_score(const T *__restrict__ q_s, const T *__restrict__ k, Call c, long long n_ctx, int n, int s_min,
             float *__restrict__ scores, int *__restrict__ done,
             int32_t *__restrict__ out_anchor, float *__restrict__ out_score) {
    extern __shared__ float dsm[];
    __shared__ int s_last;
    constexpr int E = Vec16<T>::kElems;
    constexpr int LPR = D / E;
    constexpr int RPI = 32 / LPR;
    constexpr int U = 2;
    constexpr int kWarps = kScoreThreads / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane % LPR, rsel = lane / LPR;
    const int g = blockIdx.y % c.Hkv, b = blockIdx.y / c.Hkv;
    const int h0 = g * c.G + blockIdx.z * GT;
    const long long i = n_ctx - 1;
    const T *kbase = k + b * c.kv_sb + g * c.kv_sh;

    // the attention kernel of this step may be scheduled now; it waits for this grid to finish before it reads scores.
    // This grid itself may have been launched beside the tail of the kernel before it.
    chain_release();
    chain_wait();
    float qv[GT][E];
#pragma unroll
    for (int t = 0; t < GT; ++t) Vec16<T>::load(q_s + b * c.q_sb + (long long)(h0 + t) * c.q_sh + sub * E, qv[t]);

    const int s_base = blockIdx.x * (kWarps * RPI * U);
    float part[U][GT];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int s = s_base + (u * kWarps + warp) * RPI + rsel;
#pragma unroll
        for (int t = 0; t < GT; ++t) part[u][t] = 0.f;
        if (s < n) {
            // candidate x is stride s_min + x: the first s_min strides land inside the local window
            const long long tpos = i + 1 - stride_offset(c, s_min + s);
            float kv[E];
            Vec16<T>::load(kbase + tpos * c.kv_st + sub * E, kv);
#pragma unroll
            for (int t = 0; t < GT; ++t)
#pragma unroll
                for (int e = 0; e < E; ++e) part[u][t] = fmaf(qv[t][e], kv[e], part[u][t]);
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int s = s_base + (u * kWarps + warp) * RPI + rsel;
#pragma unroll
        for (int t = 0; t < GT; ++t) {
            const float tot = reduce_sub<LPR>(part[u][t]);
            if (sub == 0 && s < n)
                scores[((long long)b * c.Hq + h0 + t) * n + s] = tot * c.search_scale;
        }
    }

    if (!done) return;   // the unsharded step selects in the attention kernel: scores only
    // ---- the CTA that completes this (batch, KV head) selects (sequence-sharded step: this rank's candidates)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const int total = gridDim.x * gridDim.z;
        const int prev = atomicAdd(done + blockIdx.y, 1);
        s_last = prev == total - 1;
        if (s_last) done[blockIdx.y] = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int per_warp = n + 2 * topk::kCap;
    float *sc = dsm + (size_t)warp * per_warp;
    float *cand_v = sc + n;
    int *cand_s = reinterpret_cast<int *>(cand_v + topk::kCap);
    for (int hg = warp; hg < c.G; hg += kWarps) {
        const long long bh = (long long)b * c.Hq + g * c.G + hg;
        const float *src = scores + bh * n;
        for (int s = lane; s < n; s += 32) sc[s] = __ldcg(src + s);   // written by other SMs: bypass L1
        __syncwarp();
        topk::select_topk(sc, n, c.top_k, i, cand_v, cand_s, out_anchor + bh * c.top_k, out_score + bh * c.top_k, lane,
                          s_min, c.off);
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------------
// Span table of one attention unit from the selected anchors (in shared memory: s_anchor[top_k], -1 = none), built
// by the whole CTA: piece starts in s_start, cumulative token counts in s_cum, the number of pieces in s_cnt (all
// visible to the CTA on return).
// Union mode: the spans of the selected anchors (Algorithm 1: S_t = [max(0,t-b l), min(i,t+f l)]) and the local
// window W = [max(0, i-w+1), i], sorted by (lo, hi) and clipped to disjoint pieces.  Per-span mode: unit j is
// J_t of the j-th selected anchor, the part of S_t left of the window and then the window; a head with nothing
// selected attends to the window alone, carried by its first unit.
// (Ranks by a ballot per interval, the intervals dealt to the warps, the clipping by prefix sums over lanes: 17
// intervals 2500 cycles; with all ranks counted by one warp through shuffles 4700.)
__device__ inline void build_unit_spans(const Call &c, long long i, long long ell, int j_unit, const int *s_anchor, int *p_lo,
                                        int *p_hi, int *s_start, int *s_cum, int *s_cnt) {
    constexpr int kWarps = kAttnThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_iv = c.top_k + (c.window > 0 ? 1 : 0);
    const int w_lo = (int)(i - c.window + 1 > 0 ? i - c.window + 1 : 0);
    auto interval = [&](int j, int &lo, int &hi) {   // absent: (INT_MAX, -1)
        lo = INT_MAX;
        hi = -1;
        if (j < c.top_k) {
            const long long t = s_anchor[j];
            if (t >= 0) {
                const long long a = t - (long long)c.back * ell, z = t + (long long)c.fwd * ell;
                lo = (int)(a > 0 ? a : 0);
                hi = (int)(z < i ? z : i);
            }
        } else if (j < n_iv) {
            lo = w_lo;
            hi = (int)i;
        }
    };
    if (c.mode == SLA_PER_SPAN) {
        if (warp == 0) {
            bool any = false;
            for (int j = lane; j < c.top_k; j += 32) any |= s_anchor[j] >= 0;
            any = __any_sync(0xffffffffu, any);
            int lo, hi;
            interval(j_unit, lo, hi);
            // a head with nothing selected attends to the window alone: its first unit carries it
            const bool sel = hi >= 0, lone_w = !any && j_unit == 0;
            const int hi_cut = c.window > 0 && hi >= w_lo ? w_lo - 1 : hi;
            const int n0 = sel && lo <= hi_cut ? hi_cut - lo + 1 : 0;
            const int n1 = (sel || lone_w) && c.window > 0 ? (int)i - w_lo + 1 : 0;
            if (lane == 0) {
                int cnt = 0;
                s_cum[0] = 0;
                if (n0) { s_start[cnt] = lo; s_cum[++cnt] = n0; }
                if (n1) { s_start[cnt] = w_lo; s_cum[cnt + 1] = n0 + n1; ++cnt; }
                *s_cnt = cnt;
            }
        }
        __syncthreads();
        return;
    }
    // rank of every interval by (lo, hi, index)
    int lo[3], hi[3];   // n_iv <= 65: intervals lane, lane + 32, lane + 64
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        lo[r] = INT_MAX;
        hi[r] = -1;
        if (32 * r < n_iv) interval(lane + 32 * r, lo[r], hi[r]);
    }
    for (int j = warp; j < n_iv; j += kWarps) {
        int lj, hj, rank = 0;
        interval(j, lj, hj);   // the same for all lanes
#pragma unroll
        for (int r = 0; r < 3; ++r)
            if (32 * r < n_iv) {
                const int m = lane + 32 * r;
                rank += __popc(__ballot_sync(0xffffffffu, m < n_iv && (lo[r] < lj || (lo[r] == lj && (hi[r] < hj || (hi[r] == hj && m < j))))));
            }
        if (lane == 0) { p_lo[rank] = lj; p_hi[rank] = hj; }
    }
    __syncthreads();
    if (warp == 0) {
        // In sorted order (absent intervals last), 32 at a time: the running maximum of the ends before an interval
        // clips its start, a prefix sum of the lengths gives the cumulative token counts, a ballot the slots of
        // the pieces that are not empty.
        int end0 = 0, cum0 = 0, cnt0 = 0;
        if (lane == 0) s_cum[0] = 0;
        for (int j0 = 0; j0 < n_iv; j0 += 32) {
            const bool on = j0 + lane < n_iv;
            const int slo = on ? p_lo[j0 + lane] : INT_MAX, shi = on ? p_hi[j0 + lane] : -1;
            int end = shi + 1;   // 0 for an absent interval
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, end, off);
                if (lane >= off) end = max(end, y);
            }
            end = max(end, end0);
            int prev_end = __shfl_up_sync(0xffffffffu, end, 1);
            if (lane == 0) prev_end = end0;
            const int start = max(slo, prev_end);
            const int len = (shi >= 0 && start <= shi) ? shi - start + 1 : 0;
            int incl = len;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            const unsigned have = __ballot_sync(0xffffffffu, len > 0);
            if (len > 0) {
                const int idx = cnt0 + __popc(have & ((1u << lane) - 1u));
                s_start[idx] = start;
                s_cum[idx + 1] = cum0 + incl;
            }
            cnt0 += __popc(have);
            cum0 += __shfl_sync(0xffffffffu, incl, 31);
            end0 = __shfl_sync(0xffffffffu, end, 31);
        }
        if (lane == 0) *s_cnt = cnt0;
    }
    __syncthreads();
}

// Top-k of sc[0..n) by the whole CTA (Section "Span search": TopK over Anchors(i)); sc[x] is the score of
// stride index s_base + x.  Result in shared memory: sel_anchor[r] / sel_score[r], r = 0 .. top_k - 1, best
// first (larger score, then the nearer anchor, i.e. the smaller stride index), padded with (-1, -inf).
//   1. the threads form at least k groups (of whole, half, ... warps); the maximum of every group is a score of its
//      own, so the smallest of the maxima is a lower bound of the k-th best score;
//   2. the scores at or above it are collected, a warp at a time (typically a few more than k);
//   3. each one's rank among them is its slot.
// When more candidates turn up than the list holds (many equal scores), every warp selects the k best of its
// eighth of the scores with the warp routine of the prefill kernels instead, and the 8 k winners are ranked.
// (1024 scores, k = 16: 7000 cycles with group maxima through shared memory and an atomic per candidate, 4300 like
// this; k rounds of a warp-wide maximum take 600 cycles each.  The loops stay rolled: the code runs once per launch,
// and fetching an instruction for the first time costs 10 to 20 cycles.)
struct SelectSmem {
    static constexpr int kCand = 256;
    alignas(16) unsigned gmax[kMaxTopK];
    int n_cand;
    alignas(16) uint2 cand[kCand];   // {order key, position in sc}
    // fallback
    float cand_v[kAttnThreads / 32][topk::kCap];
    int cand_s[kAttnThreads / 32][topk::kCap];
    int32_t anchor[kAttnThreads / 32][kMaxTopK];
    float score[kAttnThreads / 32][kMaxTopK];
};

__device__ inline void cta_select_topk(float *sc, int n, const Call &c, long long i, int s_base, SelectSmem &m, int *sel_anchor,
                                       float *sel_score) {
    constexpr int kWarps = kAttnThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = c.top_k;
    // groups of 32, 16, 8 or 4 threads: 8, 16, 32 or 64 of them
    const int gs = k <= 8 ? 32 : k <= 16 ? 16 : k <= 32 ? 8 : 4, n_groups = kAttnThreads / gs;
    // The scores are dealt to the groups in turn: no group is empty as soon as there are as many scores, however few.  (With
    // whole groups of neighbours, 90 scores filled three of eight groups, and all of them became candidates: a step of 8
    // sequences of 8191 tokens, k = 8, 37.2 to 37.7 us, and 34.4 to 36.7 us like this.)  Each turn starts at another group, so that
    // the lanes of a warp read different banks (k <= 8; two of the same for k <= 16): without that, steps of 32/4 heads were
    // up to 0.2 us longer than with neighbours (65536 tokens, k = 4: 13.90 and 13.78 us; 400000, k = 16: 58.2 and 58.1 us).
    unsigned mx = 0u;   // below every order key of a real score
    const int turn = (tid % gs) * n_groups, of_turn = (tid / gs + turn / 32) & (n_groups - 1);
#pragma unroll 1
    for (int x = turn + of_turn; x < n; x += kAttnThreads) mx = max(mx, max(topk::order_key(sc[x]), 1u));
#pragma unroll 1
    for (int off = 1; off < gs; off <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (tid % gs == 0) m.gmax[tid / gs] = mx;
    for (int j = tid; j < k; j += kAttnThreads) {
        sel_anchor[j] = -1;
        sel_score[j] = -CUDART_INF_F;
    }
    if (tid == 0) m.n_cand = 0;
    __syncthreads();
    unsigned thr = 0xffffffffu;   // 0 when some group is empty: then everything is a candidate
    for (int j = 0; j < n_groups; j += 4) {
        const uint4 g = *reinterpret_cast<const uint4 *>(m.gmax + j);
        thr = min(thr, min(min(g.x, g.y), min(g.z, g.w)));
    }
#pragma unroll 1
    for (int x0 = 0; x0 < n; x0 += kAttnThreads) {
        const int x = x0 + tid;
        const unsigned key = x < n ? max(topk::order_key(sc[x]), 1u) : 0u;
        const unsigned who = __ballot_sync(0xffffffffu, key != 0u && key >= thr);
        if (who) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&m.n_cand, __popc(who));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(who & ((1u << lane) - 1u));
            if ((who >> lane & 1u) && at < SelectSmem::kCand) m.cand[at] = make_uint2(key, (unsigned)x);
        }
    }
    __syncthreads();
    const int nc = m.n_cand;
    if (nc <= SelectSmem::kCand) {
        if (tid < nc) {
            const uint2 mine = m.cand[tid];
            int rank = 0;
#pragma unroll 2
            for (int y = 0; y < nc; ++y) {
                const uint2 o = m.cand[y];
                rank += (o.x > mine.x) || (o.x == mine.x && o.y < mine.y);
            }
            if (rank < k) {
                sel_anchor[rank] = (int)(i + 1 - stride_offset(c, s_base + (int)mine.y));
                sel_score[rank] = sc[mine.y];
            }
        }
        __syncthreads();
        return;
    }
    // ---- many equal scores: per-warp selection, then the warps' winners ranked
    const int per = (n + kWarps - 1) / kWarps;
    const int x0 = warp * per < n ? warp * per : n, x1 = x0 + per < n ? x0 + per : n;
    topk::select_topk(sc + x0, x1 - x0, k, i, m.cand_v[warp], m.cand_s[warp], m.anchor[warp], m.score[warp], lane,
                      s_base + x0, c.off);
    __syncthreads();
    for (int e = tid; e < kWarps * k; e += kAttnThreads) {
        const int w = e / k, j = e % k;
        const int a = m.anchor[w][j];
        if (a < 0) continue;
        const unsigned ka = topk::order_key(m.score[w][j]);
        int rank = 0;
        for (int w2 = 0; w2 < kWarps; ++w2)
            for (int j2 = 0; j2 < k; ++j2) {
                const int a2 = m.anchor[w2][j2];
                if (a2 < 0) break;   // a warp's winners come first, its padding last
                const unsigned k2 = topk::order_key(m.score[w2][j2]);
                rank += (k2 > ka) || (k2 == ka && a2 > a);
            }
        if (rank < k) {
            sel_anchor[rank] = a;
            sel_score[rank] = m.score[w][j];
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void cg_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cg_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }

template <typename T> __device__ __forceinline__ void unpack16(const uint4 &v, float (&f)[Vec16<T>::kElems]) {
    if constexpr (sizeof(T) == 2) {
        Vec16<__nv_bfloat16>::unpack(v, f);
    } else {
        f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
        f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
    }
}

// One attention unit per cluster row: `gridDim.x` CTAs in clusters of `cluster.num_blocks()` share a unit's tokens.
//   1. (unsharded step) the scores of the unit's head come from decode_score (`scores`), or the CTAs of a cluster score
//      a share of the anchors each and write every score to all of them; every CTA then picks the k best and builds the
//      unit's spans itself.  Sequence-sharded step: `spans` is the table decode_shard_select built.
//   2. online softmax over an even share of the tokens;
//   3. the cluster's first CTA merges the partial results of the others through distributed shared memory; when a
//      unit has several clusters, the one that finishes last merges theirs (through `partial` and the counter `done`).
// One launch or two: see the figures at plan_decode.
template <typename T, int D>
__global__ void __launch_bounds__(kAttnThreads, 2)
decode_attn(const T *__restrict__ q_s, const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, Call c,
            const int *__restrict__ spans, const float *__restrict__ scores, int n_cand, int s_min, int ell, float *__restrict__ partial, int *__restrict__ done,
            float *__restrict__ unit_out, int *__restrict__ done_head, int32_t *__restrict__ sel_anchor,
            float *__restrict__ sel_score, T *__restrict__ out, float *__restrict__ lse,
            float *__restrict__ shard_out) {
    extern __shared__ float s_scores[];   // [n_cand] (unsharded step)
    __shared__ int s_last;
    constexpr int E = Vec16<T>::kElems;
    constexpr int C = 2;                  // 16-byte chunks of a token row per lane: chunks sub and sub + LPR
    constexpr int LPR = D / (E * C);      // lanes per token row
    constexpr int RPI = 32 / LPR;
    constexpr int U = 4;
    constexpr int kWarps = kAttnThreads / 32;
    constexpr int kSlots = kWarps * RPI;  // token rows the CTA reads per load step
    constexpr int kIv = kMaxTopK + 1;
    __shared__ int s_start[kMaxTopK + 1], s_cum[kMaxTopK + 2];
    __shared__ float s_m[kSlots], s_l[kSlots];
    __shared__ float s_acc[kWarps][D];
    __shared__ int s_anchor[kMaxTopK], s_iv[2 * kIv], s_cnt;
    __shared__ float s_score[kMaxTopK];
    __shared__ SelectSmem s_sel;
    __shared__ float s_part[D + 2];         // this CTA's maximum, denominator, numerator
    cg::cluster_group cluster = cg::this_cluster();
    // the CTAs of a cluster write to each other's shared memory only when all of them have started
    if (cluster.num_blocks() > 1) cg_arrive();
    const int csize = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int sub = lane % LPR, rsel = lane / LPR;
    // attention unit: a head (union mode) or one selected anchor of a head (per-span mode)
    const bool per_span = c.mode == SLA_PER_SPAN;
    const int units = per_span ? c.top_k : 1, pcap = per_span ? 2 : c.top_k + 1;
    // (32-bit index arithmetic: at the start of a launch every instruction is fetched for the first time, about ten
    // cycles each, and a 64-bit division is a hundred of them)
    const unsigned unit32 = blockIdx.y, bh32 = per_span ? unit32 / (unsigned)units : unit32;
    const unsigned b = bh32 / (unsigned)c.Hq, h = bh32 - b * (unsigned)c.Hq, g = h / (unsigned)c.G;
    const int j_unit = (int)(unit32 - bh32 * (unsigned)units);
    const long long unit = unit32, bh = bh32;
    const int n_splits = gridDim.x, split = blockIdx.x;
    const T *kbase = k + b * c.kv_sb + g * c.kv_sh;
    const T *vbase = v + b * c.kv_sb + g * c.kv_sh;

    // launched beside the tail of the kernel before it on the stream (the score kernel, or whatever the caller runs),
    // whose results are read from here on
    chain_wait();
    int cnt;
    if (!spans) {
        const long long i = c.Lkv - 1;
        const int per = (n_cand + csize - 1) / csize, x_lo = min(rank * per, n_cand), n_loc = min(per, n_cand - x_lo);
        if (scores) {
            for (int x = tid; x < n_cand; x += kAttnThreads) s_scores[x] = __ldcg(scores + bh * n_cand + x);
        } else {
            // scores of this CTA's share of the anchors
            constexpr int LS = D / E, RS = 32 / LS, US = 4;
            const int ssub = lane % LS, srow = lane / LS;
            const uint4 q_raw = __ldg(reinterpret_cast<const uint4 *>(q_s + b * c.q_sb + (long long)h * c.q_sh + ssub * E));
            bool started = csize == 1;
#pragma unroll 1
            for (int x0 = 0; x0 < n_loc; x0 += kWarps * RS * US) {
                uint4 raw[US];
#pragma unroll
                for (int u = 0; u < US; ++u) {
                    const int x = x0 + (u * kWarps + warp) * RS + srow;
                    // candidate y is stride s_min + y: the first s_min strides land inside the local window
                    const long long t = x < n_loc ? i + 1 - stride_offset(c, s_min + x_lo + x) : i;
                    raw[u] = __ldg(reinterpret_cast<const uint4 *>(kbase + t * c.kv_st + ssub * E));
                }
                float qv[E];
                unpack16<T>(q_raw, qv);
                if (!started) cg_wait();
                started = true;
#pragma unroll
                for (int u = 0; u < US; ++u) {
                    const int x = x0 + (u * kWarps + warp) * RS + srow;
                    float kv[E], part = 0.f;
                    unpack16<T>(raw[u], kv);
#pragma unroll
                    for (int e = 0; e < E; ++e) part = fmaf(qv[e], kv[e], part);
                    part = reduce_sub<LS>(part);
                    // every CTA of the cluster gets the score: lane r of the row's lanes stores it to rank r
                    if (ssub < csize && x < n_loc) cluster.map_shared_rank(s_scores, ssub)[x_lo + x] = part * c.search_scale;
                }
            }
            if (!started) cg_wait();
        }
        if (csize > 1) cluster.sync();
        else __syncthreads();
        cta_select_topk(s_scores, n_cand, c, i, s_min, s_sel, s_anchor, s_score);
        if (split == 0 && j_unit == 0)
            for (int j = tid; j < c.top_k; j += kAttnThreads) {
                sel_anchor[bh * c.top_k + j] = s_anchor[j];
                sel_score[bh * c.top_k + j] = s_score[j];
            }
        build_unit_spans(c, i, ell, j_unit, s_anchor, s_iv, s_iv + kIv, s_start, s_cum, &s_cnt);
        cnt = s_cnt;
    } else {
        const int *sp = spans + unit * (2 * pcap + 2);
        cnt = sp[2 * pcap + 1];
        for (int j = tid; j < cnt; j += kAttnThreads) s_start[j] = sp[j];
        for (int j = tid; j <= cnt; j += kAttnThreads) s_cum[j] = sp[pcap + j];
        __syncthreads();
    }
    const long long total = cnt > 0 ? s_cum[cnt] : 0;
    const long long f_begin = total * split / n_splits, f_end = total * (split + 1) / n_splits;

    float qv[C][E];
    const float scale2 = c.softmax_scale * kLog2e;
#pragma unroll
    for (int ch = 0; ch < C; ++ch) {
        Vec16<T>::load(q + b * c.q_sb + (long long)h * c.q_sh + (ch * LPR + sub) * E, qv[ch]);
#pragma unroll
        for (int e = 0; e < E; ++e) qv[ch][e] *= scale2;
    }

    float m = -CUDART_INF_F, l = 0.f, acc[C][E];
#pragma unroll
    for (int ch = 0; ch < C; ++ch)
#pragma unroll
        for (int e = 0; e < E; ++e) acc[ch][e] = 0.f;
    int piece = 0;
    const int slot = warp * RPI + rsel;

    for (long long f0 = f_begin; f0 < f_end; f0 += kSlots * U) {
        uint4 kraw[U][C], vraw[U][C];
        bool ok[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long f = f0 + u * kSlots + slot;
            ok[u] = f < f_end;
            if (ok[u]) {
                while (f >= s_cum[piece + 1]) ++piece;
                const long long pos = s_start[piece] + (f - s_cum[piece]);
#pragma unroll
                for (int ch = 0; ch < C; ++ch) {
                    kraw[u][ch] = __ldg(reinterpret_cast<const uint4 *>(kbase + pos * c.kv_st + (ch * LPR + sub) * E));
                    vraw[u][ch] = __ldg(reinterpret_cast<const uint4 *>(vbase + pos * c.kv_st + (ch * LPR + sub) * E));
                }
            } else {
#pragma unroll
                for (int ch = 0; ch < C; ++ch) {
                    kraw[u][ch] = make_uint4(0, 0, 0, 0);
                    vraw[u][ch] = make_uint4(0, 0, 0, 0);
                }
            }
        }
        float x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x[u] = 0.f;
#pragma unroll
            for (int ch = 0; ch < C; ++ch) {
                float kv[E];
                unpack16<T>(kraw[u][ch], kv);
#pragma unroll
                for (int e = 0; e < E; ++e) x[u] = fmaf(qv[ch][e], kv[e], x[u]);
            }
        }
        float m_new = m;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x[u] = reduce_sub<LPR>(x[u]);
            if (ok[u]) m_new = fmaxf(m_new, x[u]);
        }
        const float r = (m == -CUDART_INF_F) ? 0.f : exp2f(m - m_new);
        l *= r;
#pragma unroll
        for (int ch = 0; ch < C; ++ch)
#pragma unroll
            for (int e = 0; e < E; ++e) acc[ch][e] *= r;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float p = ok[u] ? exp2f(x[u] - m_new) : 0.f;
            l += p;
#pragma unroll
            for (int ch = 0; ch < C; ++ch) {
                float vv[E];
                unpack16<T>(vraw[u][ch], vv);
#pragma unroll
                for (int e = 0; e < E; ++e) acc[ch][e] = fmaf(p, vv[e], acc[ch][e]);
            }
        }
        m = m_new;
    }

    // the next kernel may be scheduled when every CTA is here
    chain_release();
    // merge the lane groups of the warp, then the warps of the CTA
#pragma unroll
    for (int off = LPR; off < 32; off <<= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, off);
        const float ol = __shfl_xor_sync(0xffffffffu, l, off);
        const float mn = fmaxf(m, om);
        const float a = (m == -CUDART_INF_F) ? 0.f : exp2f(m - mn);
        const float bb = (om == -CUDART_INF_F) ? 0.f : exp2f(om - mn);
        l = l * a + ol * bb;
#pragma unroll
        for (int ch = 0; ch < C; ++ch)
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const float oa = __shfl_xor_sync(0xffffffffu, acc[ch][e], off);
                acc[ch][e] = acc[ch][e] * a + oa * bb;
            }
        m = mn;
    }
    if (rsel == 0) {
        if (sub == 0) { s_m[warp] = m; s_l[warp] = l; }
#pragma unroll
        for (int ch = 0; ch < C; ++ch)
#pragma unroll
            for (int e = 0; e < E; ++e) s_acc[warp][(ch * LPR + sub) * E + e] = acc[ch][e];
    }
    __syncthreads();
    if (tid < D) {
        float mm = -CUDART_INF_F;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) mm = fmaxf(mm, s_m[w]);
        float ll = 0.f, aa = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float sc = (s_m[w] == -CUDART_INF_F) ? 0.f : exp2f(s_m[w] - mm);
            ll += s_l[w] * sc;
            aa += s_acc[w][tid] * sc;
        }
        if (tid == 0) { s_part[0] = mm; s_part[1] = ll; }
        s_part[2 + tid] = aa;
    }
    float o_unit = 0.f, lse_unit = -CUDART_INF_F;
    // merge of n partial results, the x-th one found by at(x, word): {maximum, denominator, numerator[D]}
    auto merge = [&](int n, auto at, float &mm, float &ll, float &aa) {
        mm = -CUDART_INF_F;
        for (int x = 0; x < n; ++x) mm = fmaxf(mm, at(x, 0));
        ll = aa = 0.f;
        for (int x = 0; x < n; ++x) {
            const float ms = at(x, 0);
            const float sc = (ms == -CUDART_INF_F) ? 0.f : exp2f(ms - mm);
            ll += at(x, 1) * sc;
            aa += at(x, 2 + tid) * sc;
        }
    };
    float mm = -CUDART_INF_F, ll = 0.f, aa = 0.f;
    if (csize > 1) {
        cluster.sync();
        if (rank == 0 && tid < D)
            merge(csize, [&](int x, int w) { return cluster.map_shared_rank(s_part, x)[w]; }, mm, ll, aa);
        cluster.sync();   // the others' shared memory has been read
        if (rank != 0) return;
    } else {
        __syncthreads();
        if (tid < D) { mm = s_part[0]; ll = s_part[1]; aa = s_part[2 + tid]; }
    }
    const int n_clusters = n_splits / csize;
    if (n_clusters > 1) {
        // ---- the cluster that completes this unit merges the clusters' results
        if (tid < D) {
            float *dst = partial + (unit * n_clusters + split / csize) * (D + 2);
            if (tid == 0) { dst[0] = mm; dst[1] = ll; }
            dst[2 + tid] = aa;
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            const int prev = atomicAdd(done + unit, 1);
            s_last = prev == n_clusters - 1;
            if (s_last) done[unit] = 0;
        }
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (tid < D) {
            const float *src = partial + unit * n_clusters * (D + 2);
            merge(n_clusters, [&](int x, int w) { return __ldcg(src + x * (D + 2) + w); }, mm, ll, aa);
        }
    }
    if (tid < D) {
        o_unit = ll > 0.f ? aa / ll : 0.f;
        lse_unit = ll > 0.f ? (mm + log2f(ll)) * kLn2 : -CUDART_INF_F;
    }
    if (!per_span) {
        if (tid < D) {
            if (shard_out) {
                // sequence-sharded step: this rank's share of the head, merged with the others' later
                float *dst = shard_out + bh * (D + 2);
                dst[2 + tid] = o_unit;
                if (tid == 0) { dst[0] = lse_unit; dst[1] = 0.f; }
            } else {
                out[b * c.q_sb + (long long)h * c.q_sh + tid] = from_float<T>(o_unit);
                if (tid == 0) lse[bh] = lse_unit;
            }
        }
        return;
    }
    // ---- per-span mode: park A_t and its log-sum-exp; the unit that completes the head applies the gate
    if (tid < D) {
        float *dst = unit_out + unit * (D + 2);
        dst[2 + tid] = o_unit;
        if (tid == 0) dst[0] = lse_unit;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const int prev = atomicAdd(done_head + bh, 1);
        s_last = prev == units - 1;
        if (s_last) done_head[bh] = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid < D) {
        const int *an = s_anchor;      // every CTA of the head holds the head's selection
        const float *sc = s_score;
        const float *uo = unit_out + bh * units * (D + 2);
        float smax = -CUDART_INF_F;
        int n_sel = 0;
        for (int j = 0; j < c.top_k; ++j)
            if (an[j] >= 0) { smax = fmaxf(smax, sc[j]); ++n_sel; }
        float o = 0.f, l_first = -CUDART_INF_F;
        if (n_sel == 0) {
            // Algorithm 1, empty selection: the window alone (carried by the head's first unit)
            o = __ldcg(uo + 2 + tid);
            l_first = __ldcg(uo);
        } else {
            float sden = 0.f;
            for (int j = 0; j < c.top_k; ++j)
                if (an[j] >= 0) sden += expf(sc[j] - smax);
            bool first = true;
            for (int j = 0; j < c.top_k; ++j) {
                if (an[j] < 0) continue;
                o = fmaf(expf(sc[j] - smax) / sden, __ldcg(uo + j * (D + 2) + 2 + tid), o);
                if (first) { l_first = __ldcg(uo + j * (D + 2)); first = false; }
            }
        }
        out[b * c.q_sb + (long long)h * c.q_sh + tid] = from_float<T>(o);
        if (tid == 0) lse[bh] = l_first;
    }
}

// Shared memory above 48 KiB, a kernel's own 16 bytes included, has to be allowed per kernel and device context.  The score kernel
// is given the largest size it can ever be launched with, once per (device, kernel): later steps
// then launch without touching function attributes, whatever the context length.
constexpr int kScoreSmemMax = 200 * 1024;
template <auto kern>   // (by the kernel, not its type: those of all head sizes and group sizes have the same)
cudaError_t allow_score_smem(size_t smem) {
    static bool done[64] = {};
    if (smem <= 47 * 1024) return cudaSuccess;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kScoreSmemMax);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

template <typename T, int D>
cudaError_t attn_launch(const T *q_s, const T *q, const T *k, const T *v, const Call &c, const int *spans, const float *scores,
                        int n_cand, int s_min, const DecodePlan &p, int units, float *partial, int *done, float *unit_out,
                        int *done_head, int32_t *out_anchor, float *out_score, T *out, float *lse, float *shard_out,
                        cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.n_splits, c.B * c.Hq * units);
    cfg.blockDim = dim3(kAttnThreads);
    cfg.dynamicSmemBytes = (size_t)n_cand * sizeof(float);
    cfg.stream = st;
    // Programmatic dependent launch: the grid is set up while the kernel before it drains (2 to 3 us a step).  Not for
    // clusters of eight: CTAs of this grid that start in the last free slots of the one before leave the other
    // clusters no eight slots in one place (two-span steps over 1M tokens: 32 us without, 38 with it).
    cudaLaunchAttribute attr[2];
    if (p.cluster < 8) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (p.cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = p.cluster;
        attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    cfg.attrs = attr;
    return cudaLaunchKernelEx(&cfg, decode_attn<T, D>, q_s, q, k, v, c, spans, scores, n_cand, s_min,
                              (int)base_len(c, c.Lkv - 1), partial, done, unit_out,
                              done_head, out_anchor, out_score, out, lse, shard_out);
}

template <typename T, int D>
cudaError_t decode_launch(const void *q_s, const void *q, const void *k, const void *v, const Call &c,
                          long long n_ctx, const DecodePlan &p, void *scratch, int *counters, void *out, float *lse,
                          int32_t *out_anchor, float *out_score, cudaStream_t st) {
    constexpr int E = Vec16<T>::kElems;
    constexpr int RPI = 32 / (D / E);
    char *base = (char *)scratch;
    const int units = c.mode == SLA_PER_SPAN ? c.top_k : 1;
    int *done_unit = counters + c.B * c.Hkv, *done_head = done_unit + c.B * c.Hq * units;
    const int n = p.n_anchor, s_min = window_strides(c);
    const T *qs = (const T *)q_s, *kk = (const T *)k;
    if ((size_t)n * sizeof(float) > 40 * 1024) return cudaErrorInvalidValue;   // a head's scores lie in shared memory
    float *scores = nullptr;
    if (p.score_first) {
        scores = (float *)(base + p.off_scores);
        const int rows_per_cta = (kScoreThreads / 32) * RPI * 2;
        const int gt = c.G % 8 == 0 ? 8 : c.G % 4 == 0 ? 4 : c.G % 2 == 0 ? 2 : 1;
        const dim3 gs(n > 0 ? (n + rows_per_cta - 1) / rows_per_cta : 1, c.B * c.Hkv, c.G / gt);
        // scores only (no completion counter, no shared memory)
        cudaError_t e;
#define SLA_LAUNCH_SCORE(GT) \
    e = launch_chained(decode_score<T, D, GT>, gs, dim3(kScoreThreads), 0, st, qs, kk, c, n_ctx, n, s_min, scores, (int *)nullptr, \
                       out_anchor, out_score)
        switch (gt) {
            case 8: SLA_LAUNCH_SCORE(8); break;
            case 4: SLA_LAUNCH_SCORE(4); break;
            case 2: SLA_LAUNCH_SCORE(2); break;
            default: SLA_LAUNCH_SCORE(1); break;
        }
#undef SLA_LAUNCH_SCORE
        if (e != cudaSuccess) return e;
    }
    return attn_launch<T, D>(qs, (const T *)q, kk, (const T *)v, c, nullptr, scores, n, s_min, p, units,
                             (float *)(base + p.off_partial), done_unit, (float *)(base + p.off_unit_out), done_head, out_anchor,
                             out_score, (T *)out, lse, nullptr, st);
}

// ------------------------------------------------------------------------------------------------
// Sequence-sharded decode step (the KV cache of one sequence split into contiguous position ranges, one
// per rank): every rank scores the anchors that fall into its range and keeps its k best
// (decode_score without a span table); the candidates of all ranks are gathered; every rank then picks
// the global k best, clips their spans to its own range (decode_shard_select), attends to that part
// (decode_attn with a partial result) and, after a second gather, all partial results are merged through
// their log-sum-exp (decode_shard_merge).  Union mode without a local window.

// One warp per (batch, query head): global top-k of the gathered candidates (larger score first, then the
// nearer anchor, i.e. the larger position: the order of the unsharded selection) and the table of this
// rank's pieces: the spans of the selected anchors, sorted, clipped to disjoint pieces and to
// [shard_lo, shard_hi).
__global__ void __launch_bounds__(32)
decode_shard_select(const int32_t *__restrict__ all_anchor, const float *__restrict__ all_score, int n_shards,
                    Call c, long long n_ctx, long long shard_lo, long long shard_hi, int32_t *__restrict__ out_anchor,
                    float *__restrict__ out_score, int *__restrict__ spans) {
    __shared__ int s_lo[kMaxTopK], s_hi[kMaxTopK];
    const int lane = threadIdx.x;
    const long long bh = blockIdx.x, n_bh = (long long)c.B * c.Hq;
    const int k = c.top_k, n = n_shards * k;
    const long long i = n_ctx - 1;
    for (int j = lane; j < k; j += 32) {
        out_anchor[bh * k + j] = -1;
        out_score[bh * k + j] = -CUDART_INF_F;
    }
    __syncwarp();
    for (int x = lane; x < n; x += 32) {
        const long long src = ((long long)(x / k) * n_bh + bh) * k + x % k;
        const int ax = all_anchor[src];
        if (ax < 0) continue;
        const uint32_t kx = topk::order_key(all_score[src]);
        int rank = 0;
        for (int y = 0; y < n; ++y) {
            const long long sy = ((long long)(y / k) * n_bh + bh) * k + y % k;
            const int ay = all_anchor[sy];
            if (ay < 0) continue;
            const uint32_t ky = topk::order_key(all_score[sy]);
            rank += (ky > kx) || (ky == kx && ay > ax);
        }
        if (rank < k) {
            out_anchor[bh * k + rank] = ax;
            out_score[bh * k + rank] = all_score[src];
        }
    }
    __syncwarp();
    if (lane == 0) {
        // spans of the selected anchors (Algorithm 1: S_t = [max(0,t-b l), min(i,t+f l)]), insertion-sorted
        const long long ell = base_len(c, i);
        int m = 0;
        for (int j = 0; j < k; ++j) {
            const long long t = out_anchor[bh * k + j];
            if (t < 0) continue;
            const long long a = t - (long long)c.back * ell, z = t + (long long)c.fwd * ell;
            const int l0 = (int)(a > 0 ? a : 0), h0 = (int)(z < i ? z : i);
            int pos = m;
            while (pos > 0 && (s_lo[pos - 1] > l0 || (s_lo[pos - 1] == l0 && s_hi[pos - 1] > h0))) {
                s_lo[pos] = s_lo[pos - 1];
                s_hi[pos] = s_hi[pos - 1];
                --pos;
            }
            s_lo[pos] = l0;
            s_hi[pos] = h0;
            ++m;
        }
        const int pcap = k + 1;
        int *start = spans + bh * (2 * pcap + 2);
        int *cum = start + pcap;
        int cnt = 0;
        long long next_free = 0, total = 0;
        cum[0] = 0;
        for (int a = 0; a < m; ++a) {
            long long j0 = s_lo[a] > next_free ? s_lo[a] : next_free;
            if ((long long)s_hi[a] + 1 > next_free) next_free = (long long)s_hi[a] + 1;
            // this rank's part of the piece
            long long j1 = s_hi[a];
            if (j0 < shard_lo) j0 = shard_lo;
            if (j1 > shard_hi - 1) j1 = shard_hi - 1;
            if (j0 <= j1) {
                start[cnt] = (int)j0;
                total += j1 - j0 + 1;
                cum[cnt + 1] = (int)total;
                ++cnt;
            }
        }
        start[2 * pcap + 1] = cnt;
    }
}

// One CTA per (batch, query head): merge of the ranks' partial results {lse, -, o[D]} (fp32).
template <typename T, int D>
__global__ void __launch_bounds__(D)
decode_shard_merge(const float *__restrict__ all_partial, int n_shards, Call c, T *__restrict__ out,
                   float *__restrict__ lse) {
    const long long bh = blockIdx.x, n_bh = (long long)c.B * c.Hq;
    const int h = (int)(bh % c.Hq), b = (int)(bh / c.Hq), tid = threadIdx.x;
    float mm = -CUDART_INF_F;
    for (int w = 0; w < n_shards; ++w) mm = fmaxf(mm, all_partial[((long long)w * n_bh + bh) * (D + 2)]);
    float den = 0.f, acc = 0.f;
    if (mm > -CUDART_INF_F) {
        for (int w = 0; w < n_shards; ++w) {
            const float *src = all_partial + ((long long)w * n_bh + bh) * (D + 2);
            if (src[0] == -CUDART_INF_F) continue;
            const float wt = expf(src[0] - mm);
            den += wt;
            acc = fmaf(wt, src[2 + tid], acc);
        }
    }
    out[b * c.q_sb + (long long)h * c.q_sh + tid] = from_float<T>(den > 0.f ? acc / den : 0.f);
    if (tid == 0) lse[bh] = den > 0.f ? mm + logf(den) : -CUDART_INF_F;
}

template <typename T, int D>
cudaError_t shard_search_launch(const void *q_s, const void *k_local, const Call &c, long long n_ctx, int s_first,
                                int n, void *scratch, int *counters, int32_t *cand_anchor, float *cand_score,
                                cudaStream_t st) {
    constexpr int E = Vec16<T>::kElems;
    constexpr int RPI = 32 / (D / E);
    float *scores = (float *)scratch;
    const int rows_per_cta = (kScoreThreads / 32) * RPI * 2;
    const int gt = c.G % 8 == 0 ? 8 : c.G % 4 == 0 ? 4 : c.G % 2 == 0 ? 2 : 1;
    dim3 gs(n > 0 ? (n + rows_per_cta - 1) / rows_per_cta : 1, c.B * c.Hkv, c.G / gt);
    // positions are global: the local slice starts at shard_lo
    const T *qs = (const T *)q_s, *kk = (const T *)k_local - c.shard_lo * c.kv_st;
    const size_t smem = (size_t)(kScoreThreads / 32) * (n + 2 * topk::kCap) * sizeof(float);
    if (smem > (size_t)kScoreSmemMax) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
#define SLA_LAUNCH_SCORE(GT)                                                                                         \
    do {                                                                                                             \
        constexpr auto kern = decode_score<T, D, GT>;                                                                \
        e = allow_score_smem<kern>(smem);                                                                            \
        if (e == cudaSuccess)                                                                                        \
            kern<<<gs, kScoreThreads, smem, st>>>(qs, kk, c, n_ctx, n, s_first, scores, counters, cand_anchor,       \
                                                  cand_score);                                                      \
    } while (0)
    switch (gt) {
        case 8: SLA_LAUNCH_SCORE(8); break;
        case 4: SLA_LAUNCH_SCORE(4); break;
        case 2: SLA_LAUNCH_SCORE(2); break;
        default: SLA_LAUNCH_SCORE(1); break;
    }
#undef SLA_LAUNCH_SCORE
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <typename T, int D>
cudaError_t shard_attend_launch(const void *q, const void *k_local, const void *v_local, const Call &c, long long n_ctx,
                                const DecodePlan &p, void *scratch, int *counters, int n_shards,
                                const int32_t *all_anchor, const float *all_score, int32_t *out_anchor,
                                float *out_score, float *partial_out, cudaStream_t st) {
    char *base = (char *)scratch;
    int *spans = (int *)(base + p.off_spans);
    float *partial = (float *)(base + p.off_partial);
    int *done_unit = counters + c.B * c.Hkv, *done_head = done_unit + c.B * c.Hq;
    decode_shard_select<<<c.B * c.Hq, 32, 0, st>>>(all_anchor, all_score, n_shards, c, n_ctx, c.shard_lo, c.shard_hi,
                                                   out_anchor, out_score, spans);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const T *kk = (const T *)k_local - c.shard_lo * c.kv_st, *vv = (const T *)v_local - c.shard_lo * c.kv_st;
    DecodePlan ps = p;
    ps.cluster = 1;
    return attn_launch<T, D>(nullptr, (const T *)q, kk, vv, c, spans, nullptr, 0, 0, ps, 1, partial, done_unit, nullptr, done_head, out_anchor,
                             out_score, nullptr, nullptr, partial_out, st);
}

}  // namespace

#define SLA_DISPATCH(fn, ...)                                                                    \
    (dtype == SLA_F32 ? (c.D == 64 ? fn<float, 64>(__VA_ARGS__) : fn<float, 128>(__VA_ARGS__))   \
                      : (c.D == 64 ? fn<__nv_bfloat16, 64>(__VA_ARGS__) : fn<__nv_bfloat16, 128>(__VA_ARGS__)))

cudaError_t launch_decode_shard_search(const void *q_s, const void *k_local, const Call &c, int dtype,
                                       long long n_ctx, int s_first, int n, void *scratch, int *counters,
                                       int32_t *cand_anchor, float *cand_score, cudaStream_t st) {
    return SLA_DISPATCH(shard_search_launch, q_s, k_local, c, n_ctx, s_first, n, scratch, counters, cand_anchor,
                        cand_score, st);
}

cudaError_t launch_decode_shard_attend(const void *q, const void *k_local, const void *v_local, const Call &c,
                                       int dtype, long long n_ctx, const DecodePlan &plan, void *scratch,
                                       int *counters, int n_shards, const int32_t *all_anchor,
                                       const float *all_score, int32_t *out_anchor, float *out_score,
                                       float *partial_out, cudaStream_t st) {
    return SLA_DISPATCH(shard_attend_launch, q, k_local, v_local, c, n_ctx, plan, scratch, counters, n_shards,
                        all_anchor, all_score, out_anchor, out_score, partial_out, st);
}

cudaError_t launch_decode_shard_merge(const float *all_partial, int n_shards, const Call &c, int dtype, void *out,
                                      float *lse, cudaStream_t st) {
    const unsigned grid = (unsigned)(c.B * c.Hq);
    if (dtype == SLA_F32) {
        if (c.D == 64) decode_shard_merge<float, 64><<<grid, 64, 0, st>>>(all_partial, n_shards, c, (float *)out, lse);
        else decode_shard_merge<float, 128><<<grid, 128, 0, st>>>(all_partial, n_shards, c, (float *)out, lse);
    } else {
        if (c.D == 64)
            decode_shard_merge<__nv_bfloat16, 64><<<grid, 64, 0, st>>>(all_partial, n_shards, c, (__nv_bfloat16 *)out, lse);
        else
            decode_shard_merge<__nv_bfloat16, 128><<<grid, 128, 0, st>>>(all_partial, n_shards, c, (__nv_bfloat16 *)out, lse);
    }
    return cudaGetLastError();
}
#undef SLA_DISPATCH


int decode_attn_blocks_per_sm(int dtype, int D) {
    // resident CTAs per SM with the shared memory a 16M-token context needs for a head's anchor scores
    constexpr size_t kOccSmem = 16 * 1024;
    static int cache[2][2] = {{0, 0}, {0, 0}};
    int &slot = cache[dtype == SLA_F32 ? 0 : 1][D == 64 ? 0 : 1];
    if (slot == 0) {
        int n = 0;
        cudaError_t e;
        if (dtype == SLA_F32)
            e = D == 64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, decode_attn<float, 64>, kAttnThreads, kOccSmem)
                        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, decode_attn<float, 128>, kAttnThreads, kOccSmem);
        else
            e = D == 64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, decode_attn<__nv_bfloat16, 64>, kAttnThreads, kOccSmem)
                        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, decode_attn<__nv_bfloat16, 128>, kAttnThreads, kOccSmem);
        slot = (e == cudaSuccess && n > 0) ? n : 1;
    }
    return slot;
}

constexpr int kShare = 128;   // anchors per CTA that it scores itself

DecodePlan plan_decode(const Call &c, long long n_ctx, int cta_slots, size_t gap) {
    DecodePlan p;
    // candidates: the strides whose anchor lies left of the local window
    const long long n_cand = n_strides(c, n_ctx - 1) - window_strides(c);
    p.n_anchor = (int)(n_cand > 0 ? n_cand : 0);
    const long long ell = base_len(c, n_ctx - 1);
    long long span_tokens = (long long)(c.back + c.fwd) * ell + 1;
    if (span_tokens > n_ctx) span_tokens = n_ctx;
    const bool per_span = c.mode == SLA_PER_SPAN;
    const int units = per_span ? c.top_k : 1, pcap = per_span ? 2 : c.top_k + 1;
    const long long win = c.window < n_ctx ? c.window : n_ctx;
    const long long max_tokens = per_span ? span_tokens + win : span_tokens * c.top_k + win;
    // one resident wave: as many splits per attention unit as fit the CTA slots of the device
    long long ns = (long long)cta_slots / ((long long)c.B * c.Hq * units);
    if (ns > max_tokens / 128) ns = max_tokens / 128;
    if (ns > 256) ns = 256;
    if (ns < 1) ns = 1;
    // One launch, the CTAs of a unit in clusters (the largest power of two up to 8) that share the scoring and the
    // merge, or two, all scores first.  One launch saves the score kernel and its hand-over (8 sequences of 8191
    // tokens 45 -> 36 us, a two-span step over 100003 tokens 28.7 -> 23.5), but a CTA scores its share after its start
    // (7 us for 400 anchors: 16 x 181104 tokens 272 -> 280), so the share is bounded; and splits beyond the clusters
    // are left idle (8 of 9 per head at 1M tokens: 92 -> 100 us), which may cost 24 MB of reading at most, the time
    // that is saved.
    const int csz = ns >= 8 ? 8 : ns >= 4 ? 4 : ns >= 2 ? 2 : 1, fused = (int)(ns / csz) * csz;
    const long long bytes = (long long)c.B * c.Hq * units * max_tokens * 2 * c.D * 2;
    const bool one = p.n_anchor <= csz * kShare && (double)bytes * (ns - fused) / ns < 24e6;
    p.score_first = !one;
    p.cluster = one ? csz : 1;
    p.n_splits = one ? fused : (int)ns;
    const size_t bh = (size_t)c.B * c.Hq, n_units = bh * units;
    size_t off = 0;
    // a region of `size` bytes at the next 256-byte boundary, with a canary gap before it when asked for
    auto take = [&](size_t size) {
        if (gap) { p.canaries.add(off); off += gap; }
        const size_t at = off;
        off = (off + size + 255) & ~(size_t)255;
        return at;
    };
    p.off_scores = take(bh * (size_t)p.n_anchor * sizeof(float));
    p.off_spans = take(n_units * (size_t)(2 * pcap + 2) * sizeof(int));
    p.off_partial = take(n_units * (size_t)p.n_splits * (c.D + 2) * sizeof(float));
    p.off_unit_out = take(per_span ? n_units * (size_t)(c.D + 2) * sizeof(float) : 0);
    if (gap) { p.canaries.add(off); off += gap; }
    p.bytes = off;
    return p;
}

cudaError_t launch_decode(const void *q_s, const void *q, const void *k, const void *v, const Call &c,
                          int dtype, long long n_ctx, const DecodePlan &plan, void *scratch, int *counters,
                          void *out, float *lse, int32_t *out_anchor, float *out_score, cudaStream_t st) {
    if (dtype == SLA_F32) {
        return c.D == 64 ? decode_launch<float, 64>(q_s, q, k, v, c, n_ctx, plan, scratch, counters, out, lse, out_anchor, out_score, st)
                         : decode_launch<float, 128>(q_s, q, k, v, c, n_ctx, plan, scratch, counters, out, lse, out_anchor, out_score, st);
    }
    return c.D == 64 ? decode_launch<__nv_bfloat16, 64>(q_s, q, k, v, c, n_ctx, plan, scratch, counters, out, lse, out_anchor, out_score, st)
                     : decode_launch<__nv_bfloat16, 128>(q_s, q, k, v, c, n_ctx, plan, scratch, counters, out, lse, out_anchor, out_score, st);
}

// ------------------------------------------------------------------------------------------------
// Decode step for callers that cannot allocate device memory (declared in include/sla.h).
//
// Some hosts of this library run where cudaMalloc is off limits: inside a CUDA-graph capture or a
// stream-ordered region of a serving loop, in a process whose device memory is handed out in full to
// another allocator at start-up, or in a plug-in that is only lent a stream.  They cannot create an
// sla handle (its workspace is a cudaMalloc).  For them the decode step's scratch -- anchor scores,
// clipped spans, split results and the completion counters -- lives in the array below, which is
// part of the library image: every GPU that loads the library holds these 2 MiB until the process
// exits, whether or not the entry point is ever called.
namespace {

constexpr size_t kStaticScratchBytes = SLA_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_decode_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
// Device addresses of the array, one per device.  In host code the array's name is only a handle for
// the runtime: the address a kernel may use comes from cudaGetSymbolAddress, asked once per device
// with that device current.
unsigned char *g_decode_scratch_ptr[kMaxDevices] = {};
int g_cta_slots[kMaxDevices][2][2] = {};

}  // namespace
}  // namespace sla

extern "C" sla_status_t sla_decode_step_static(const void *q_s, const void *q, const void *k_cache,
                                               const void *v_cache, int64_t n_ctx, const sla_layout_t *l,
                                               const sla_params_t *p, void *out, float *lse, int32_t *out_anchor,
                                               float *out_score, void *stream) {
    sla::Call c;
    if (sla_status_t s = sla::check_decode_args(q_s, q, k_cache, v_cache, n_ctx, l, p, out, lse, out_anchor, out_score, &c))
        return s;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SLA_ERR_CUDA;
    if (dev < 0 || dev >= sla::kMaxDevices) return SLA_ERR_UNSUPPORTED;
    if (!sla::g_decode_scratch_ptr[dev]) {
        // set-up, once per device (the current one): resolve the array's device address
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, sla::g_decode_scratch) != cudaSuccess || !ptr) return SLA_ERR_CUDA;
        sla::g_decode_scratch_ptr[dev] = static_cast<unsigned char *>(ptr);
    }
    int &slots = sla::g_cta_slots[dev][l->dtype == SLA_F32 ? 0 : 1][l->head_dim == 64 ? 0 : 1];
    if (slots == 0) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return SLA_ERR_CUDA;
        slots = sms * sla::decode_attn_blocks_per_sm(l->dtype, l->head_dim);
    }
    const sla::DecodePlan plan = sla::plan_decode(c, n_ctx, slots);
    const size_t counter_bytes = (((size_t)l->batch * (l->n_kv_heads + l->n_q_heads) * sizeof(int)) + 255) & ~(size_t)255;
    if (counter_bytes + plan.bytes > sla::kStaticScratchBytes) return SLA_ERR_WORKSPACE;   // beyond the fixed maximum
    if ((size_t)plan.n_anchor * sizeof(float) * 8 > 180 * 1024) return SLA_ERR_UNSUPPORTED;
    unsigned char *base = sla::g_decode_scratch_ptr[dev];
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the array keeps whatever the previous call left; only the completion counters have to start at zero
    if (cudaMemsetAsync(base, 0, counter_bytes, st) != cudaSuccess) return SLA_ERR_CUDA;
    cudaError_t e = sla::launch_decode(q_s, q, k_cache, v_cache, c, l->dtype, n_ctx, plan, base + counter_bytes,
                                       reinterpret_cast<int *>(base), out, lse, out_anchor, out_score, st);
    return e == cudaSuccess ? SLA_OK : SLA_ERR_CUDA;
}
