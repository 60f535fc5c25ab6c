// Work-list construction for the tensor-core span-attention kernel: a counting sort of all pieces
// (clipped spans) of a chunk of query rows by (batch*Hkv + kv head, 64-key block of the piece's
// right end, class of blocks covered), and the table of 256-piece tiles cut from the sorted list.
//
// This is the step Section "Kernel design" describes as grouping (query, span) pairs into buckets by
// key-block footprint without a global sort.  Each CTA owns a slice of the rows of one
// (batch, kv head), counts its pieces in a shared-memory histogram and touches the global counters
// once per non-empty bucket, so that global atomics stay far below one per piece.
//
//   prep_clear       bucket counts and cursors to zero
//   prep_count       the pieces of every row, parked; histogram of bucket sizes; pieces per row
//   prep_scan        per (batch, kv head): exclusive offsets of its buckets, record and tile totals
//   prep_scatter     the parked pieces to their places in the sorted list; tile table entries (a tile = 256
//                    consecutive records of the sorted list, whatever end blocks they fall in)
//   prep_tile_bounds per tile: split where neighbouring pieces end far apart; the tile's end block and how
//                    far back its pieces reach (number of key blocks to walk)
#include <limits.h>

#include "sla_attn_tc.cuh"

namespace sla {
namespace tc {

namespace {

constexpr int kPrepThreads = 1024;
// Without being asked the runtime gives a kernel 48 KB of shared memory, its own arrays included (128 bytes at most beside a histogram).
constexpr size_t kPlainSmem = 47 * 1024;
constexpr size_t kMostSmem = kHistBytes + kMaxWalk + 16;   // histogram and class table of the longest list
static_assert(kMostSmem <= 226 * 1024, "a CTA has 227 KB");

// Bucket of a piece: its end block and the class of the number of blocks it covers.  Classes are even
// steps over [0, nb_single) (a single span) and, for joined pieces, over [nb_single, nb_max).
__device__ __forceinline__ int class_of(int len, const PrepArgs &a) {
    int cls;
    if (len < a.nb_single || a.ncls == a.ncls1) {
        cls = (len * a.ncls1) / a.nb_single;
        cls = cls < a.ncls1 ? cls : a.ncls1 - 1;
    } else {
        cls = a.ncls1 + ((len - a.nb_single) * (a.ncls - a.ncls1)) / (a.nb_max - a.nb_single + 1);
        cls = cls < a.ncls ? cls : a.ncls - 1;
    }
    return cls;
}
// Classes run upwards in even end blocks and downwards in odd ones, so that the sorted list changes
// length smoothly from one end block to the next (tiles are cut across those boundaries).
__device__ __forceinline__ int bucket_at(int eb, int cls, const PrepArgs &a) {
    return eb * a.ncls + ((eb & 1) ? a.ncls - 1 - cls : cls);
}
__device__ __forceinline__ int bucket_of(int lo, int hi, const PrepArgs &a) {
    const int eb = hi / kBK, sb = lo / kBK;
    return bucket_at(eb, class_of(eb - sb, a), a);
}

// Union-mode pieces of one row for at most K intervals (anchors + window), streamed: emit(lo, hi, n) is
// called for the n-th piece, left to right.  Same pieces as row_pieces up to the order in which
// intervals with the same left end are clipped (the union, and with it the attention, is the same).
// All spans of a row are equally long before clipping, so ordering them by anchor orders them by
// (lo, hi); the window W = [w_lo, i] takes its place through the anchor that would give lo = w_lo.
// Keys are 2t for a span and 2t_W + 1 for W (after the spans that start at or before w_lo).
template <int K, typename Emit>
__device__ __forceinline__ int union_pieces_stream(const int32_t *__restrict__ an, int top_k, int i, long long ell,
                                                   int back, int fwd, int window, int merge_cap, int *status,
                                                   Emit emit) {
    constexpr unsigned kAbsent = 0xffffffffu;
    const long long bl64 = (long long)back * ell, fl64 = (long long)fwd * ell;
    const int bl = bl64 > INT_MAX ? INT_MAX : (int)bl64, fl = fl64 > INT_MAX ? INT_MAX : (int)fl64;
    const int w_lo = i - window + 1 > 0 ? i - window + 1 : 0;
    unsigned key[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        key[j] = kAbsent;
        if (j < top_k) {
            const int t = an[j];
            if (t > i) atomicOr(status, kStatusBadIndex);
            else if (t >= 0) key[j] = 2u * (unsigned)t;
        } else if (j == top_k && window > 0) {
            unsigned tw = (unsigned)w_lo + (unsigned)bl;
            if (tw > (unsigned)i + 1u) tw = (unsigned)i + 1u;
            if (tw > 0x7ffffffeu) tw = 0x7ffffffeu;   // stays below the "absent" key
            key[j] = 2u * tw + 1u;
        }
    }
#pragma unroll
    for (int round = 0; round < K; ++round)
#pragma unroll
        for (int x = round & 1; x + 1 < K; x += 2) {
            const unsigned lo_ = min(key[x], key[x + 1]), hi_ = max(key[x], key[x + 1]);
            key[x] = lo_;
            key[x + 1] = hi_;
        }
    int cnt = 0, cur_lo = 0, cur_hi = -1, next_free = 0;
    bool have = false;
#pragma unroll
    for (int x = 0; x < K; ++x) {
        const unsigned kx = key[x];
        const bool present = kx != kAbsent;
        const int t = (int)(kx >> 1);
        int l0, h0;
        if (kx & 1u) {
            l0 = w_lo;
            h0 = i;
        } else {
            l0 = bl >= t ? 0 : t - bl;
            h0 = fl >= i - t ? i : t + fl;
        }
        const int j0 = l0 > next_free ? l0 : next_free;
        const bool on = present && j0 <= h0;
        // the piece in hand ends at next_free - 1: an interval that continues right there is joined to it
        const bool join = on && have && j0 == next_free && h0 - cur_lo < merge_cap;
        if (on && !join) {
            if (have) emit(cur_lo, cur_hi, cnt++);
            cur_lo = j0;
            have = true;
        }
        if (on) cur_hi = h0;
        if (present && h0 + 1 > next_free) next_free = h0 + 1;
    }
    if (have) emit(cur_lo, cur_hi, cnt++);
    return cnt;
}

// Rows of one (batch, kv head) are shared out evenly among ctas_per_bg CTAs, the same way in both passes.
struct Share {
    int bg, g, b;
    long long q0, q1;
};
__device__ __forceinline__ Share share_of(const PrepArgs &a) {
    Share s;
    s.bg = blockIdx.x / a.ctas_per_bg;
    const int part = blockIdx.x % a.ctas_per_bg;
    s.g = s.bg % a.Hkv;
    s.b = s.bg / a.Hkv;
    const long long rows_bg = (long long)a.G * a.Lc;
    const long long per = (rows_bg + a.ctas_per_bg - 1) / a.ctas_per_bg;
    s.q0 = per * part < rows_bg ? per * part : rows_bg;   // a CTA beyond the last row gets an empty range
    s.q1 = (s.q0 + per < rows_bg) ? s.q0 + per : rows_bg;
    return s;
}
__device__ __forceinline__ int row_of(const PrepArgs &a, const Share &s, long long q, int &h, int &rc) {
    const int hg = (int)((unsigned)q / (unsigned)a.Lc);   // G * Lc < 2^31
    rc = (int)((unsigned)q % (unsigned)a.Lc);
    h = s.g * a.G + hg;
    return (int)(((long long)s.b * a.Hq + h) * a.Lc + rc);
}

// Where a CTA parks the n-th piece of its row q: all first pieces, then all second ones, ...  A warp's rows are neighbours, so that
// it writes and reads whole sectors, and the slots that no row fills are never touched.  65536 positions, 32/8 heads, eight spans:
// counting pass 162 us with a row's pieces side by side, 95 like this, scatter pass 172 and 147; 16384 33 and 25, 27 and 24 (ncu).
__device__ __forceinline__ int4 *parked(const PrepArgs &a, const Share &s, long long q, int n) {
    const long long row0 = ((long long)s.b * a.Hq + s.g * a.G) * a.Lc + s.q0;   // the CTA's rows are consecutive
    return a.stage + row0 * a.slots + n * (s.q1 - s.q0) + (q - s.q0);
}

// Counting pass.  Every piece of the CTA's rows is built once, counted in the CTA's shared-memory
// histogram (the value the atomic returns is the piece's ordinal within its bucket and CTA) and parked
// in `stage`; the histogram goes to the global bucket counts and, whole, to cta_hist.
// K: compile-time bound on the intervals of a row (anchors + window) for the register-resident piece
// builder, or 0 for the general one.
template <int K>
__global__ void __launch_bounds__(kPrepThreads) prep_count(PrepArgs a) {
    extern __shared__ int hist[];   // [NB * ncls]
    constexpr int KA = K > 0 ? K : kMaxTopK + 1;
    const int nk = a.NB * a.ncls;
    const Share sh = share_of(a);
    // class of every "blocks covered" value, behind the histogram
    unsigned char *cls_tbl = reinterpret_cast<unsigned char *>(hist + nk);
    for (int x = threadIdx.x; x < nk; x += kPrepThreads) hist[x] = 0;
    for (int x = threadIdx.x; x <= a.nb_max; x += kPrepThreads) cls_tbl[x] = (unsigned char)class_of(x, a);
    __syncthreads();
    chain_wait();
    chain_release();
    int lo[KA], hi[KA], slot[KA];
    for (long long q = sh.q0 + threadIdx.x; q < sh.q1; q += kPrepThreads) {
        int h, rc;
        const int row = row_of(a, sh, q, h, rc);
        const long long r = a.r0 + rc, i = a.q_pos0 + r;
        const int32_t *an = a.anchor + (((long long)sh.b * a.Hq + h) * a.Lq + r) * a.top_k;
        const long long ell = base_len(i, a.span_len, a.len_first, a.n_len);
        if constexpr (K > 0) {
            if (a.mode == SLA_UNION) {
                int4 *st = parked(a, sh, q, 0);
                const long long pitch = sh.q1 - sh.q0;
                const int n = union_pieces_stream<KA>(an, a.top_k, (int)i, ell, a.back, a.fwd, a.window, a.merge_cap, a.status,
                                                      [&](int l0, int h0, int ordinal) {
                                                          const int eb = h0 / kBK, len = eb - l0 / kBK;
                                                          const int bucket = bucket_at(eb, cls_tbl[len < a.nb_max ? len : a.nb_max], a);
                                                          const int ord = atomicAdd(&hist[bucket], 1);
                                                          st[ordinal * pitch] = make_int4(l0, h0, bucket | (ordinal << 24), ord);
                                                      });
                a.n_pieces[row] = (unsigned char)n;
                continue;
            }
        }
        int cnt;
        if constexpr (K > 0)
            cnt = row_pieces_per_span_small<KA>(an, a.top_k, i, ell, a.back, a.fwd, a.window, lo, hi, slot, a.status);
        else
            cnt = row_pieces(an, a.top_k, i, ell, a.back, a.fwd, a.window, a.mode, a.merge_cap, lo, hi, slot, a.status);
        a.n_pieces[row] = (unsigned char)cnt;
        int4 *st = parked(a, sh, q, 0);
        const long long pitch = sh.q1 - sh.q0;
        auto park = [&](int j) {
            const int bucket = bucket_of(lo[j], hi[j], a);
            const int ord = atomicAdd(&hist[bucket], 1);
            st[j * pitch] = make_int4(lo[j], hi[j], bucket | (slot[j] << 24), ord);
        };
        if constexpr (K > 0) {
#pragma unroll
            for (int j = 0; j < KA; ++j)
                if (j < cnt) park(j);
        } else {
            for (int j = 0; j < cnt; ++j) park(j);
        }
    }
    __syncthreads();
    int *gcount = a.key_count + (long long)sh.bg * nk;
    int *mine = a.cta_hist + (long long)blockIdx.x * nk;
    for (int x = threadIdx.x; x < nk; x += kPrepThreads) {
        const int c = hist[x];
        mine[x] = c;
        if (c) atomicAdd(gcount + x, c);
    }
}

// Scatter pass: the CTA claims a contiguous range of every bucket it has pieces in (its count is in
// cta_hist, the bucket's offset within its (batch, kv head) in key_count by now) and moves its parked pieces to
// their places.
// kFewRows: at most kFewScatter rows a CTA, several threads a row.  With a thread a row few threads went through up to 65 pieces each and the
// others had none: 16 positions of 32/8 heads, 64 spans 12.2 and 5.7 us; 300 positions, 8/2 heads 14.8 and 6.3; 1200 (267 rows a CTA) 19.2
// and 17.4 (ncu).  Not where a thread moves a row's pieces in one step, nor with two threads a row: 2000 positions, 64 spans 5.4 and 6.4 us.
// (An instantiation of its own: in one kernel the other lists' pass took 48 registers instead of 32 and 1999 positions, four spans 0.2 to 0.4 us more.)
constexpr int kScatterStep = 4;   // pieces a thread has in flight
constexpr int kFewScatter = kPrepThreads / 3;   // three threads a row at least
template <bool kFewRows>
__global__ void __launch_bounds__(kPrepThreads) prep_scatter(PrepArgs a) {
    extern __shared__ int hist[];   // [NB * ncls]: first record of this CTA in every bucket
    const int nk = a.NB * a.ncls;
    const Share sh = share_of(a);
    const int *gcount = a.key_count + (long long)sh.bg * nk;
    int *gcursor = a.key_cursor + (long long)sh.bg * nk;
    const int *mine = a.cta_hist + (long long)blockIdx.x * nk;
    __shared__ int s_base[2];   // records and tiles of the (batch, kv head)s before this one
    chain_wait();
    chain_release();
    if (threadIdx.x < 32) {
        int recs = 0, tiles = 0;
        for (int x = threadIdx.x; x < sh.bg; x += 32) {
            recs += a.totals[2 * x];
            tiles += a.totals[2 * x + 1];
        }
        recs = __reduce_add_sync(0xffffffffu, recs);
        tiles = __reduce_add_sync(0xffffffffu, tiles);
        if (threadIdx.x == 0) {
            s_base[0] = recs;
            s_base[1] = tiles;
        }
    }
    // four buckets per thread and round, so that the counts, then the claims, are in flight together
    for (int x0 = threadIdx.x; x0 < nk; x0 += 4 * kPrepThreads) {
        int cnt[4], first[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int x = x0 + u * kPrepThreads;
            cnt[u] = x < nk ? mine[x] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int x = x0 + u * kPrepThreads;
            first[u] = cnt[u] ? gcount[x] + atomicAdd(gcursor + x, cnt[u]) : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int x = x0 + u * kPrepThreads;
            if (x < nk) hist[x] = first[u];
        }
    }
    __syncthreads();
    const int rec_base = s_base[0];
    if (blockIdx.x == sh.bg * a.ctas_per_bg) {
        // the first CTA of the (batch, kv head) cuts its part of the sorted list into tiles of kRows records, across end blocks:
        // entries {batch*Hkv + kv head, (end block: filled in by prep_tile_bounds), first record, records}
        const int n_recs = a.totals[2 * sh.bg], nt = a.totals[2 * sh.bg + 1], tile_base = s_base[1];
        for (int t = threadIdx.x; t < nt; t += kPrepThreads) {
            const int left = n_recs - t * kRows;
            if (tile_base + t < a.max_tiles)
                a.tiles[tile_base + t] = make_int4(sh.bg, 0, rec_base + t * kRows, left < kRows ? left : kRows);
        }
        if (sh.bg == a.B * a.Hkv - 1 && threadIdx.x == 0) {
            const int all = tile_base + nt;
            a.n_tiles[0] = a.n_tiles[1] = all < a.max_tiles ? all : a.max_tiles;   // [1]: the count as cut here
            a.n_tiles[2] = 0;   // tiles claimed by the attention kernel
        }
    }
    // One thread per row, four pieces in flight per thread; the last rows first, whose pieces the L2 still holds.
    constexpr int U = kScatterStep;
    const int n_rows = (int)(sh.q1 - sh.q0);
    const int row_base = (int)(((long long)sh.b * a.Hq + sh.g * a.G) * a.Lc + sh.q0);   // rows x slots < 2^31 for the whole chunk
    const int4 *st = parked(a, sh, sh.q0, 0);
    if constexpr (kFewRows) {
        // as many threads as there are for each row, the slots read along with the number of pieces (one beyond it holds stale bytes
        // that are not looked at)
        if (n_rows == 0) return;
        const int sharers = kPrepThreads / n_rows, part = (int)threadIdx.x / n_rows, ql = n_rows - 1 - ((int)threadIdx.x - part * n_rows);
        if (part >= sharers) return;
        const int cnt = a.n_pieces[row_base + ql];
        for (int j0 = part * U, end = a.slots; j0 < end; j0 += sharers * U, end = cnt) {
            int4 pc[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 + u < end) pc[u] = __ldg(st + (long long)(j0 + u) * n_rows + ql);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 + u < cnt)
                    a.recs[rec_base + hist[pc[u].z & 0xffffff] + pc[u].w] = make_int4(row_base + ql, pc[u].z >> 24, pc[u].x, pc[u].y);
        }
        return;
    }
    int ql = n_rows - 1 - (int)threadIdx.x;
    int cnt = ql >= 0 ? a.n_pieces[row_base + ql] : 0;
    for (; ql >= 0;) {
        const int next = ql - kPrepThreads, next_cnt = next >= 0 ? a.n_pieces[row_base + next] : 0;
        for (int j0 = 0; j0 < cnt; j0 += U) {
            int4 pc[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 + u < cnt) pc[u] = __ldg(st + (long long)(j0 + u) * n_rows + ql);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 + u < cnt)
                    a.recs[rec_base + hist[pc[u].z & 0xffffff] + pc[u].w] = make_int4(row_base + ql, pc[u].z >> 24, pc[u].x, pc[u].y);
        }
        ql = next;
        cnt = next_cnt;
    }
}

// Exclusive scan over the block: returns this thread's offset, total in `total`.
__device__ inline int block_excl_scan(int v, int &total, int *warp_sum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = warp_sum[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        warp_sum[lane] = w;
    }
    __syncthreads();
    total = warp_sum[31];
    const int base = warp > 0 ? warp_sum[warp - 1] : 0;
    __syncthreads();
    return base + x - v;
}

// The bucket counts and cursors start from zero.
__global__ void __launch_bounds__(kPrepThreads) prep_clear(PrepArgs a) {
    const long long n = (long long)a.B * a.Hkv * a.NB * a.ncls;
    const long long x0 = (long long)blockIdx.x * 4 * kPrepThreads + threadIdx.x;
    chain_wait();
    chain_release();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const long long x = x0 + u * kPrepThreads;
        if (x < n) a.key_count[x] = a.key_cursor[x] = 0;
    }
}

// One CTA per (batch, kv head): bucket histogram -> exclusive offsets local to the (batch, kv head),
// plus how many records and tiles it has.  Many buckets lie in shared memory meanwhile: read and written whole lines at a time, an
// odd number per thread, so that the threads of a warp read different banks.  Each thread's own straight from global memory, and
// like this (ncu): 14336 buckets 23.8 and 12.4 us, 40960 41.7 and 13.3, but 8192 6.4 and 7.5.
constexpr int kScanDirect = 8;   // buckets per thread that are read straight from global memory
template <bool kShared>
__global__ void __launch_bounds__(kPrepThreads) prep_scan(PrepArgs a) {
    extern __shared__ int hist[];   // kShared: [NB * ncls]
    __shared__ int warp_sum[32];
    const int nk = a.NB * a.ncls, bg = blockIdx.x, tid = threadIdx.x;
    int *cnt = a.key_count + (long long)bg * nk, *at = kShared ? hist : cnt;
    const int most = (nk + kPrepThreads - 1) / kPrepThreads, per = kShared ? most | 1 : most;
    const int k0 = per * tid < nk ? per * tid : nk, k1 = (k0 + per < nk) ? k0 + per : nk;
    chain_wait();
    chain_release();
    if constexpr (kShared) {
#pragma unroll 8
        for (int k = tid; k < nk; k += kPrepThreads) hist[k] = cnt[k];
        __syncthreads();
    }
    int local = 0;
    for (int k = k0; k < k1; ++k) local += at[k];
    int n_recs;
    int run = block_excl_scan(local, n_recs, warp_sum);
    for (int k = k0; k < k1; ++k) {
        const int c = at[k];
        at[k] = run;
        run += c;
    }
    if constexpr (kShared) {
        __syncthreads();
        for (int k = tid; k < nk; k += kPrepThreads) cnt[k] = hist[k];
    }
    // tiles: the sorted list of the (batch, kv head) is cut every kRows records, across end blocks
    if (tid == 0) {
        a.totals[2 * bg] = n_recs;
        a.totals[2 * bg + 1] = (n_recs + kRows - 1) / kRows;
    }
}

// One warp per tile as cut by prep_scatter (256 consecutive records).  Where two neighbouring records of the
// tile end further apart than a span is long the tile is split there: walking the gap would cost more than walking
// two spans.  Where few rows look into a long context a tile's records may lie far apart without such a gap, and one CTA
// would walk them all from end to end: in a list of fewer than kSplitTiles tiles per CTA a tile is also split into
// stretches of end blocks, a power of two between one and a half and three times a span's length (each part walks a span
// more; parts of less than 2^kMinStretch blocks would not hide the gather of their Q rows).  In other lists stretches of
// 2^kMaxStretch blocks keep the block numbers of a tile within 16 bits.
// Search and attention, without and with that split: 182 rows of 32/8 heads at 123447, one span of 703 keys and a window
// of 1088 724 and 286 us; 69 rows of 16/8 heads at 195044, four spans of 1765 keys 881 and 368 us; 417 rows of 8/2 heads at 246543,
// 17 spans of 373 keys 304 and 290 us.
// The extra tiles are appended to the table.  For every tile: the end block of its last piece (second word), the
// number of key blocks from the one its furthest-reaching piece starts in up to that end block (bits 9.. of the last
// word), and the part of that walk each stream of 128 pieces reaches (`ranges`).
constexpr int kSplitTiles = 3;
constexpr int kMinStretch = 4, kMaxStretch = 14;
__global__ void __launch_bounds__(256) prep_tile_bounds(PrepArgs a) {
    __shared__ int s_eb[8][kRows], s_lo[8][kRows];
    __shared__ unsigned s_cut[8][kRows / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * 8 + warp;
    chain_wait();
    chain_release();
    if (t >= a.n_tiles[1]) return;
    const int4 ti = a.tiles[t];
    const int cnt = ti.w, shift = a.n_tiles[1] < kSplitTiles * a.ctas ? max(kMinStretch, 31 - __clz(3 * a.nb_single)) : kMaxStretch;
    int *eb = s_eb[warp], *lo = s_lo[warp];
    for (int x = lane; x < cnt; x += 32) {
        const int4 rec = a.recs[ti.z + x];
        eb[x] = rec.w / kBK;
        lo[x] = rec.z;
    }
    __syncwarp();
    // the records a part starts at: beyond a gap (records are ordered by end block), or in another stretch than the one
    // before it; the parts but the first take their places in the table together
    int n_extra = 0, extra = 0;
    if (eb[cnt - 1] - eb[0] > a.nb_single) {
#pragma unroll 1
        for (int w = 0; w < kRows / 32; ++w) {
            const int x = 32 * w + lane;
            const bool cut = x > 0 && x < cnt && (eb[x] - eb[x - 1] > a.nb_single || (eb[x] - eb[0]) >> shift != (eb[x - 1] - eb[0]) >> shift);
            const unsigned m = __ballot_sync(0xffffffffu, cut);
            if (lane == 0) s_cut[warp][w] = m;
            n_extra += __popc(m);
        }
        __syncwarp();
        if (n_extra > 0) {
            if (lane == 0) extra = atomicAdd(a.n_tiles, n_extra);
            extra = __shfl_sync(0xffffffffu, extra, 0);
        }
    }
    int seg0 = 0, idx = t;
    while (seg0 < cnt) {
        int seg1 = cnt;
        for (int w = (seg0 + 1) / 32; n_extra > 0 && w < kRows / 32; ++w) {
            const unsigned m = s_cut[warp][w] & (w == (seg0 + 1) / 32 ? ~0u << ((seg0 + 1) % 32) : ~0u);
            if (m) {
                seg1 = 32 * w + __ffs(m) - 1;
                break;
            }
        }
        // the two streams of 128 pieces: what each reaches, and the tile's walk that covers both
        const int mid = min(seg0 + kRows / 2, seg1);
        int lo_a = INT_MAX, lo_b = INT_MAX;
        for (int x = seg0 + lane; x < seg1; x += 32) {
            if (x < mid) lo_a = min(lo_a, lo[x]);
            else lo_b = min(lo_b, lo[x]);
        }
        lo_a = __reduce_min_sync(0xffffffffu, lo_a);
        lo_b = __reduce_min_sync(0xffffffffu, lo_b);
        const int eb_last = eb[seg1 - 1], sb = min(lo_a, lo_b) / kBK;
        if (lane == 0) {
            if (idx < a.max_tiles) {
                a.tiles[idx] = make_int4(ti.x, eb_last, ti.z + seg0, (seg1 - seg0) | ((eb_last - sb + 1) << 9));
                a.ranges[idx] = make_int2((lo_a / kBK - sb) | ((eb[mid - 1] - sb + 1) << 16),
                                          mid < seg1 ? (lo_b / kBK - sb) | ((eb_last - sb + 1) << 16) : 0);
            } else
                atomicOr(a.status, kStatusBadIndex);   // cannot happen: the table has room for one tile per bucket more
        }
        seg0 = seg1;
        idx = extra++;
    }
}

}  // namespace

cudaError_t prepare(const PrepArgs &a, cudaStream_t st, long long *launches) {
    const int n_bg = a.B * a.Hkv;
    // histogram, and behind it the class table of the counting pass (one byte per length)
    const size_t smem = (size_t)a.NB * a.ncls * sizeof(int) + (((size_t)a.nb_max + 1 + 15) & ~(size_t)15);
    // register-resident piece builder for up to 5 / 9 / 17 anchors and window together, the general one otherwise (search and
    // attention with 9 and with 5 entries: 1999 positions, four spans 100.3 and 98.8 us; 1590 positions, two 44.5 and 43.4 us)
    const int n_iv = a.top_k + (a.window > 0 ? 1 : 0);
    const int variant = n_iv <= 5 ? 3 : n_iv <= 9 ? 0 : n_iv <= 17 ? 1 : 2;
    void (*k0)(PrepArgs) = variant == 3 ? prep_count<5> : variant == 0 ? prep_count<9> : variant == 1 ? prep_count<17> : prep_count<0>;
    const bool few = a.slots > kScatterStep && ((long long)a.G * a.Lc + a.ctas_per_bg - 1) / a.ctas_per_bg <= kFewScatter;
    void (*k1)(PrepArgs) = few ? prep_scatter<true> : prep_scatter<false>;
    const bool many = a.NB * a.ncls > kScanDirect * kPrepThreads;
    const size_t scan_smem = many ? (size_t)a.NB * a.ncls * sizeof(int) : 0;
    // Function attributes belong to a device's context: remembered per device.  A kernel is given the most that any list takes, so that
    // no later call or other thread has to raise it, or lowers it.
    static bool allowed[64][7] = {};   // the four counting kernels, the two scatter kernels and the scan
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    const bool known = dev >= 0 && dev < 64;
    auto allow = [&](void (*kern)(PrepArgs), int which, size_t bytes) -> cudaError_t {
        if (bytes <= kPlainSmem || (known && allowed[dev][which])) return cudaSuccess;
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMostSmem);
        if (e == cudaSuccess && known) allowed[dev][which] = true;
        return e;
    };
    cudaError_t e = allow(k0, variant, smem);
    if (e == cudaSuccess) e = allow(k1, 4 + few, smem);
    if (e == cudaSuccess) e = allow(prep_scan<true>, 6, scan_smem);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)(n_bg * a.ctas_per_bg);
    // a chain of short kernels: 1999 positions, 32/8 heads, search to merge, 115 us with plain launches, a memset and an
    // extra kernel for the offsets across (batch, kv head)s, 101 us like this; 16/2 heads, 1590 positions, K = 2 61 and 46 us
    const long long words = (long long)n_bg * a.NB * a.ncls;
    const unsigned clear = (unsigned)((words + 4 * kPrepThreads - 1) / (4 * kPrepThreads));
    e = launch_chained(prep_clear, dim3(clear), dim3(kPrepThreads), 0, st, a);
    if (e == cudaSuccess) e = launch_chained(k0, dim3(grid), dim3(kPrepThreads), smem, st, a);
    if (e == cudaSuccess) e = launch_chained(many ? prep_scan<true> : prep_scan<false>, dim3(n_bg), dim3(kPrepThreads), scan_smem, st, a);
    if (e == cudaSuccess) e = launch_chained(k1, dim3(grid), dim3(kPrepThreads), smem, st, a);
    if (e == cudaSuccess) e = launch_chained(prep_tile_bounds, dim3((unsigned)((a.max_tiles + 7) / 8)), dim3(256), 0, st, a);
    if (launches) *launches += 5;
    return e;
}

}  // namespace tc
}  // namespace sla
