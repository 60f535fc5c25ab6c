// Tensor-core span-attention for prefill (bf16, head_dim 128): tcgen05 MMA with TMEM accumulators,
// K/V tiles by TMA, one softmax thread per query row.
//
// What it computes is Section "Span attention" (A_{i,t} = Attention(Q(i), K[S_t], V[S_t])) with the
// spans of Algorithm 1.  Union mode: the k spans of a (query, head) row (and its local window) are
// sorted and clipped to disjoint "pieces"; every piece is attended on its own and the per-piece
// results are merged exactly through their log-sum-exp.  Per-span mode (Algorithm 1 literally): the
// pieces are the spans themselves (the part left of the window) plus the window once per row; the
// merge forms every A_t from its span piece and the window piece and applies the gate of Section
// "Combination".
//
// The systems problem (Section "Kernel design"): neighbouring queries pick different spans, so the
// rows of one MMA tile must be made to share a key footprint.  Here pieces are grouped by the
// 64-key block their right end falls in (per batch and KV head) and, inside a group, ordered by how
// many key blocks they cover, with one counting sort (histogram, prefix sum, scatter) -- no
// comparison sort of the queries.  A tile is 256 consecutive pieces of the sorted list (of one group,
// or of neighbouring groups whose end blocks lie next to each other), two streams of 128: their Q rows are
// gathered into shared memory and the tile walks the key blocks they cover from left to right.
//
//   tc::prepare          the counting sort and the tile table (sla_attn_prep.cu)
//   tc_attend            persistent CTAs; tiles are claimed in the order of the table (short lists and short
//                        walks: tile t goes to CTA t mod grid); per tile and key block: S = Q K^T (tcgen05, smem x smem -> TMEM), row
//                        softmax in registers, P (bf16) back into TMEM, O += P V (tcgen05, TMEM x smem
//                        -> TMEM); per piece a normalised fp16 block-floating-point partial + lse
//   tc_merge             per row: log-sum-exp merge of its pieces -> out, lse
//   tc_merge_gated       per row: A_t = merge(span piece, window piece), O = sum_t alpha_t A_t
//
// CTA layout of tc_attend (512 threads, one CTA per SM): warps 0-3 and 4-7 are the softmax warps of the
// tile's two streams (one thread per piece, TMEM lane = row); warps 8-11 write the results (and gather the
// first tile's Q and, where the tiles are dealt, the second stream's); warps 12 and 13 issue the MMAs of a stream each; warp 14
// loads K and V, once for both streams; warp 15 claims the tiles to come and gathers their Q.  TMEM: per stream 128 columns of O and two 64-column S
// buffers (P aliases the S it came from).  Every wait on an mbarrier is bounded; when one runs out the CTA
// raises a status bit, drains and leaves.
//
// What bounds it: a stream's chain per 64-key block (S ready -> softmax -> P -> PV, S two blocks ahead), the
// special-function pipe (1024 cycles of exponentials for a block of both streams) and the tensor pipe (1376: an
// N = 64 S instruction holds it for 52 cycles, not 32, for its operand traffic); it takes about 1950 cycles.
// Before, two independent CTAs per SM of 128 pieces each, whose row threads also gathered Q and wrote results:
// 1860 cycles a block in long tiles but 5300 more per tile; now 700 per tile.  Configuration of 65536 tokens, 11
// blocks per tile: 4.07 -> 3.45 ms; 16384 tokens, 7 blocks: 658 -> 570 us.
// Two things that the times depend on: the kernel's code has to fit the instruction cache (sm__icc_request_hit_rate at 16384
// positions: 99.8 % dealt, 99.5 % claiming; a larger variant that was 5 % slower had 93 %), and the issuing warps have to
// run converged with one elected lane issuing (see ptx::elect_one): the issuers' time per block bounded the
// streams at 2500 cycles otherwise.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <limits.h>
#include <math_constants.h>
#include <stddef.h>

#include "sla_attn_tc.cuh"
#include "sla_tc_ptx.cuh"

namespace sla {

namespace {

using bf16 = __nv_bfloat16;

constexpr int kD = 128;
using tc::kBK;    // keys per block of the work list
using tc::kRows;  // pieces per tile
using tc::kMaxWalk;
constexpr int kHalf = 128;       // pieces per stream: a tile's first and second 128
constexpr int kThreads = 512;    // 4 row warps per stream, 4 epilogue warps, an MMA issuer per stream, K/V producer, Q gather
constexpr int kTmemCols = 512;
constexpr int kMinTiles = 1024;  // entries of the tile table at least: more than CTAs
constexpr uint32_t kColO = 0;    // O of the streams at columns 0 and 128
constexpr uint32_t kColS = 256;  // two S buffers of 64 columns per stream, from columns 256 and 384; P aliases its S
constexpr int kQBytes = kHalf * kD * 2;      // 32 KiB, two 64-wide halves of 128 rows x 128 B
constexpr int kKVBytes = kBK * kD * 2;       // 16 KiB, two 64-wide halves of 64 rows x 128 B
constexpr int kQS = 4;           // Q buffers: two per stream, in turn (buffer 2 * (n & 1) + x for the n-th tile of stream x)
constexpr int kKS = 3;           // K and V stages
constexpr int kTS = 4;           // entries of the ring of tiles
// A list is claimed tile by tile if it can have kClaimTiles tiles per CTA (every slot of every row taken) and its longest single
// piece, a span or the window, can cover kClaimBlocks key blocks (kClaimBlocksJoined where touching spans are joined, which
// makes the walks longer).  Dealt round-robin, the CTAs of a long list end at different times: SMs were busy for 0.87 of the
// kernel at 16384 positions and 0.94 at 65536, and are for 0.95 and 0.97 claimed (553 and 521 us; 3569 and 3491 us).  Tiles of short
// walks lose more by the claims than by that.  The kernel, 32/8 heads, eight spans, dealt and claimed, us (runs of one side differ by 1 to 5 %):
//   joined, from position 0    16384, spans of 65 / 129 / 193 / 257 keys (3 / 4 / 5 / 6 blocks)
//                                                597, 658 / 590, 628 / 667, 651 / 735, 707
//                              65536, the same   2529, 2828 / 2752, 2812 / 2950, 2926 / 3593, 3119
//                              4736, 257 keys 178, 173;  9000, 301 keys 432, 387
//   not joined, at 90000       12000, spans of 193 / 321 / 385 / 513 keys (5 / 7 / 8 / 10 blocks)
//                                                551, 642 / 705, 751 / 824, 822 / 977, 920
//   per span, 32768            four spans of 257 keys, window 256 (6 blocks) 965, 994; spans of 65, window 1088 (18) 1553, 1402
//   tiles per CTA, at 100000, spans of 635 keys (11 blocks): 5: 183, 185; 7: 200, 206; 12: 245, 241; 16: 302, 282; 40: 593, 589
// Joined lists have fewer tiles than the slots of their rows suggest.  With walks this long either side wins by the way its
// tiles happen to fall, up to 18 % (16 spans of 513 keys at 4736, 7 tiles per CTA: 255, 279; eight of them 274, 232).
constexpr int kClaimTiles = 16, kClaimBlocks = 8, kClaimBlocksJoined = 5;
// They are read by one lane each of the row and epilogue warps, whose waits are answered for the whole warp, and by every
// lane of the issuers and of the K/V producer, whose lanes wait each for itself (a vote in each of their waits made the
// kernel 1 % slower at 16384 positions).
constexpr int kTileReaders = 12 + 3 * 32;
constexpr int kOffQ = 0;
constexpr int kOffK = kQS * kQBytes;
constexpr int kOffV = kOffK + kKS * kKVBytes;
constexpr int kOffMeta = kOffV + kKS * kKVBytes;   // 229376
constexpr int kMetaBytes = 3072;
constexpr int kSmemBytes = kOffMeta + kMetaBytes;  // 227 KiB: one CTA per SM
constexpr float kRescaleThreshold = 8.f;     // log2 units: P stays below 2^8
// registers per thread after the re-split; the sum over the four warpgroups stays within the 4 x 128 of the launch
constexpr int kRegsRow = 160, kRegsEpi = 96, kRegsIssue = 96;
static_assert(2 * kRegsRow + kRegsEpi + kRegsIssue <= 4 * 128, "more registers than the block is launched with");

struct Meta {
    unsigned long long q_full[kQS], q_empty[kQS], kv_full[kKS], kv_empty[2][kKS];
    unsigned long long s_full[4], p_ready[4], l_full[2], o_full[2], o_empty[2], t_full[kTS], t_empty[kTS];
    uint32_t tmem_base;
    int abort_flag;
    int4 tile[kTS];        // the CTA's tiles: table entry (no records: none is left) and the blocks its streams reach
    int2 range[kTS];
    float2 stats[kRows];   // {reciprocal denominator, log2-domain log-sum-exp} of the tile's rows, for the epilogue
};
static_assert(sizeof(Meta) <= kMetaBytes, "meta block too large");

struct TcParams {
    const bf16 *q;             // Q as rows at one pitch (in elements), numbered as in its tensor map
    long long q_pitch;
    int q_b, q_h, q_t;         // strides of Q in those rows
    int Hq, Lc, slots;         // slots: partial results per row (top_k, + 1 with a local window)
    int r0;                    // first query row of the chunk
    float scale2;              // softmax_scale * log2(e)
    int slot_t, slot_h, slot_b;  // positions of (token, head, batch) among tensor-map coordinates 1..3
    const int4 *recs;          // sorted piece records {row, j, lo, hi}
    const int4 *tiles;         // {b*Hkv+g, end block, first record, record count | key blocks to walk << 9}
    const int2 *ranges;        // key blocks of the walk a tile's streams take part in: first | end << 16
    int *n_tiles;              // number of tiles; [2]: tiles claimed beyond the first two of every CTA
    __half *part_o;            // [rows*slots][128] normalised piece outputs, fp16 with one power-of-two
                               // scale per 32-column chunk (block floating point)
    float2 *part_lse;          // [rows*slots] {log2-domain log-sum-exp of the piece, four chunk exponents}
    int *status;
    int Hkv;
};

// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// packed fp32x2 arithmetic (two independent fp32 lanes per instruction)
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long r, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ unsigned long long ffma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long fadd2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// A shared-memory matrix descriptor moved forward by `bytes` (the start address sits in the low word
// in units of 16 bytes, and the window is far below the field's range, so no carry leaves it).
__device__ __forceinline__ uint64_t desc_advance(uint64_t desc, uint32_t bytes) {
    uint32_t lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(desc));
    lo += bytes >> 4;
    asm("mov.b64 %0, {%1, %2};" : "=l"(desc) : "r"(lo), "r"(hi));
    return desc;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// kClaim: tiles beyond a CTA's first two are claimed when they are needed, else dealt round-robin.
template <bool kClaim>
__global__ void __launch_bounds__(kThreads, 1)
tc_attend(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
          const __grid_constant__ CUtensorMap tm_v, TcParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t base = ptx::smem_u32(smem);
    Meta *meta = reinterpret_cast<Meta *>(smem + kOffMeta);
    volatile int *abort_flag = &meta->abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (base & 1023u) {   // the swizzled tiles need a 1024-byte aligned window: refuse rather than corrupt
        if (tid == 0) atomicOr(p.status, kStatusTimeout);
        return;
    }
    const uint32_t mbase = base + kOffMeta;
    const uint32_t bar_q_full = mbase + offsetof(Meta, q_full), bar_q_empty = mbase + offsetof(Meta, q_empty);
    const uint32_t bar_kv_full = mbase + offsetof(Meta, kv_full), bar_kv_empty = mbase + offsetof(Meta, kv_empty);
    const uint32_t bar_s_full = mbase + offsetof(Meta, s_full), bar_p_ready = mbase + offsetof(Meta, p_ready);
    const uint32_t bar_l_full = mbase + offsetof(Meta, l_full);
    const uint32_t bar_o_full = mbase + offsetof(Meta, o_full), bar_o_empty = mbase + offsetof(Meta, o_empty);
    const uint32_t bar_t_full = mbase + offsetof(Meta, t_full), bar_t_empty = mbase + offsetof(Meta, t_empty);

    if (tid == 0) {
#pragma unroll 1
        for (int x = 0; x < kQS; ++x) {
            // an arrival of each epilogue warp, or that of the gather and three of the same lane beside it
            ptx::mbar_init(bar_q_full + 8 * x, 4);
            ptx::mbar_init(bar_q_empty + 8 * x, 1);
        }
#pragma unroll 1
        for (int x = 0; x < kKS; ++x) {
            ptx::mbar_init(bar_kv_full + 8 * x, 1);
            ptx::mbar_init(bar_kv_empty + 8 * x, 1);
            ptx::mbar_init(bar_kv_empty + 8 * (kKS + x), 1);
        }
#pragma unroll 1
        for (int x = 0; x < 4; ++x) {
            ptx::mbar_init(bar_s_full + 8 * x, 1);
            ptx::mbar_init(bar_p_ready + 8 * x, 4);   // one arrival per row warp
            static_assert(kTS == 4, "the ring's barriers are initialised with those of the four S buffers");
            ptx::mbar_init(bar_t_full + 8 * x, 1);
            ptx::mbar_init(bar_t_empty + 8 * x, kTileReaders);
        }
#pragma unroll 1
        for (int x = 0; x < 2; ++x) {
            ptx::mbar_init(bar_l_full + 8 * x, 4);
            ptx::mbar_init(bar_o_full + 8 * x, 1);
            ptx::mbar_init(bar_o_empty + 8 * x, 4);
        }
        meta->abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 12) {
        ptx::tmem_alloc(mbase + offsetof(Meta, tmem_base), kTmemCols);
        ptx::tmem_relinquish();
    }
    // the set-up above runs beside the kernel before this one
    chain_wait();
    chain_release();
    const int n_tiles = *p.n_tiles;
    // the role's tile; no records when none is left.  (The table has an entry for every CTA.)
    int4 ti = p.tiles[blockIdx.x];
    int2 rg;                          // blocks of its walk the streams take part in
    // The ring's first entry.  Every role has read the table's already and takes only the range; without the store of the other
    // half, though, the per-span mode took 0.3 to 0.6 % longer, as with a loop of its own for the ring's barriers above.
    if (kClaim && tid == 0) {
        meta->tile[0] = ti;
        meta->range[0] = p.ranges[blockIdx.x];
        ptx::mbar_arrive(bar_t_full);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = meta->tmem_base;
    if (blockIdx.x >= n_tiles) ti = make_int4(0, 0, 0, 0);   // not an entry: nothing below looks records up through it
    auto first_range = [&]() { return ti.w ? (kClaim ? meta->range[0] : p.ranges[blockIdx.x]) : make_int2(0, 0); };

    constexpr uint32_t kIdescS = ptx::idesc_bf16_f32(kHalf, kBK, false, false);   // S = Q K^T, both K-major
    constexpr uint32_t kIdescO = ptx::idesc_bf16_f32(kHalf, kD, false, true);       // O = P V, V is N-major

    // Off the critical path the claiming kernel uses the shorter form of the waits, for the instruction cache.
    auto wait_aside = [&](uint32_t bar, uint32_t parity) {
        if constexpr (kClaim) return ptx::mbar_wait_short(bar, parity, abort_flag);
        else return ptx::mbar_wait(bar, parity, abort_flag);
    };
    // The first two tiles of CTA c are c and c + grid of the table.  The warp that gathers Q claims the others, in the order of the
    // table, and passes each one's entry {b*Hkv+g, end block, first record, count | blocks << 9} on through a ring in shared
    // memory; a list that is not claimed is dealt round-robin, and every role reads the table itself.
    auto read_tile = [&](uint32_t k) {   // the CTA's k-th tile; every lane gets its own answer
        if constexpr (kClaim) {
            const bool got = ptx::mbar_wait_short(bar_t_full + 8 * (k % kTS), (k / kTS) & 1u, abort_flag);
            ti = meta->tile[k % kTS];
            rg = meta->range[k % kTS];
            return got;
        } else {
            const int n = blockIdx.x + k * gridDim.x;
            ti = n < n_tiles ? p.tiles[n] : make_int4(0, 0, 0, 0);
            rg = n < n_tiles ? p.ranges[n] : make_int2(0, 0);
            return true;
        }
    };
    auto lane_read = [&](uint32_t k) {   // the lane needs the entry no more
        if constexpr (kClaim) ptx::mbar_arrive(bar_t_empty + 8 * (k % kTS));
    };
    // The same for a whole warp.  Not in the issuers and the K/V producer: there a lane whose wait ran out leaves alone, and
    // the others would wait for it here without a bound.
    auto warp_read = [&](uint32_t k) {
        if constexpr (kClaim) {
            __syncwarp();
            if (lane == 0) lane_read(k);
        }
    };
    auto take_tile = [&](uint32_t k) {
        const bool got = __all_sync(0xffffffffu, read_tile(k));
        warp_read(k);
        return got;
    };
    auto q_row = [&](int row, int bb) {   // number of a record's row among the rows of Q
        const int bh = (unsigned)row / (unsigned)p.Lc;
        return bb * p.q_b + (bh - bb * p.Hq) * p.q_h + (p.r0 + row - bh * p.Lc) * p.q_t;
    };

    if (warp >= 12) {
        ptx::setmaxnreg_dec<kRegsIssue>();
        if (warp < 14) {
            // ---------------- MMA issuer of stream x: a whole warp, its elected lane issues.  Block after block, across
            // tile boundaries, S runs two blocks ahead of PV: S(n+2) reuses the buffer of P(n) and is issued right
            // behind PV(n) (the tensor pipe keeps a thread's order).  The first PV of a tile overwrites O, so it waits
            // until the epilogue has read the tile before.  Blocks that none of the stream's pieces reach are only
            // handed on.  Two waits and two commits per block: the issuer's own time per block bounds the stream.
            const bool leader = ptx::elect_one();
            const int x = warp - 12;
            struct Cursor {
                uint32_t k;       // tile
                int j, nblk;      // nblk 0: no tile left
                int first, end;   // blocks this stream takes part in
                uint32_t nb;      // of those so far
            };
            auto open = [&](Cursor &c) {   // the tile just read
                const int r = x ? rg.y : rg.x;
                c.j = 0;
                c.nblk = ti.w >> 9;
                c.first = r & 0xffff;
                c.end = r >> 16;
            };
            Cursor cs{0u, 0, 0, 0, 0, 0u};
            rg = first_range();
            open(cs);
            Cursor cv = cs;
            bool ok = true;
            const uint32_t s_col = tmem + kColS + x * (2 * kBK), o_col = tmem + kColO + x * kD;
            uint32_t nq = 0, t = 0;   // tiles of the stream that S and PV are through with
            const uint64_t desc_q0 = ptx::smem_desc_sw128(base + kOffQ, 16, 1024);
            const uint64_t desc_k0 = ptx::smem_desc_sw128(base + kOffK, 16, 1024);
            const uint64_t desc_v0 = ptx::smem_desc_sw128(base + kOffV, kKVBytes / 2, 1024);
#pragma unroll 1
            for (uint32_t i = 0; ok && cv.nblk > 0; ++i) {
                if (i >= 2) {
                    const uint32_t st = (i - 2) % kKS, bar_done = bar_kv_empty + 8 * (x * kKS + st);
                    const bool last = cv.j == cv.end - 1;
                    if (cv.j >= cv.first && cv.j < cv.end) {
                        const uint32_t b = cv.nb & 1u;
                        if (cv.j == cv.first && t > 0 && !ptx::mbar_wait(bar_o_empty + 8 * x, (t - 1u) & 1u, abort_flag)) break;
                        if (!ptx::mbar_wait(bar_p_ready + 16 * x + 8 * b, (cv.nb >> 1) & 1u, abort_flag)) break;
                        ptx::tc_fence_after();
                        const uint64_t dv = desc_advance(desc_v0, st * kKVBytes);
                        if (leader) {
#pragma unroll
                            for (int kk = 0; kk < kBK / 16; ++kk)
                                ptx::mma_ts(o_col, s_col + b * kBK + kk * 8, desc_advance(dv, kk * 2048), kIdescO, cv.j - cv.first + kk);
                            ptx::mma_commit(bar_done);
                            if (last) ptx::mma_commit(bar_o_full + 8 * x);
                        }
                        ++cv.nb;
                        t += last;
                    } else if (leader) {
                        ptx::mbar_arrive(bar_done);
                    }
                    if (++cv.j == cv.nblk) {
                        ok = read_tile(++cv.k);   // S has opened it before
                        open(cv);
                    }
                }
                if (ok && cs.nblk > 0) {
                    const uint32_t st = i % kKS;
                    if (!ptx::mbar_wait(bar_kv_full + 8 * st, (i / kKS) & 1u, abort_flag)) break;
                    const bool last = cs.j == cs.end - 1;
                    if (cs.j >= cs.first && cs.j < cs.end) {
                        const uint32_t qs = 2 * (nq & 1u) + x, b = cs.nb & 1u;
                        if (cs.j == cs.first && !ptx::mbar_wait(bar_q_full + 8 * qs, (nq >> 1) & 1u, abort_flag)) break;
                        ptx::tc_fence_after();
                        const uint64_t dq = desc_advance(desc_q0, qs * kQBytes), dk = desc_advance(desc_k0, st * kKVBytes);
                        if (leader) {
#pragma unroll
                            for (int kk = 0; kk < kD / 16; ++kk)
                                ptx::mma_ss(s_col + b * kBK, desc_advance(dq, (kk >> 2) * (kQBytes / 2) + (kk & 3) * 32),
                                            desc_advance(dk, (kk >> 2) * (kKVBytes / 2) + (kk & 3) * 32), kIdescS, kk > 0);
                            ptx::mma_commit(bar_s_full + 16 * x + 8 * b);
                            if (last) ptx::mma_commit(bar_q_empty + 8 * qs);
                        }
                        ++cs.nb;
                        nq += last;
                    }
                    if (++cs.j == cs.nblk) {
                        ok = read_tile(++cs.k);
                        open(cs);
                    }
                }
                // a tile that PV has left is given back behind the S, which the row warps may be waiting for: 32 arrivals
                // of a lane each (two sequences of 262144 positions 94.9 ms a call with them before it, 94.5 like this)
                if (cv.j == 0 && cv.k > 0) lane_read(cv.k - 1);
            }
        } else if (warp == 14) {
            // ---------------- K/V producer: K and V of block after block, each as two halves of the head dimension
            const bool leader = ptx::elect_one();
            uint32_t n = 0, k = 0;
            bool ok = true;
            lane_read(0);
            while (ok && ti.w) {
                const int nblk = ti.w >> 9, bb = (unsigned)ti.x / (unsigned)p.Hkv, t0 = (ti.y + 1 - nblk) * kBK;
                int c[4];
                c[1 + p.slot_h] = ti.x - bb * p.Hkv;
                c[1 + p.slot_b] = bb;
                ok = read_tile(++k);
                lane_read(k);
#pragma unroll 1
                for (int j = 0; j < nblk && ok; ++j, ++n) {
                    const uint32_t st = n % kKS, ph = ((n / kKS) & 1u) ^ 1u;
                    c[1 + p.slot_t] = t0 + j * kBK;
                    ok = wait_aside(bar_kv_empty + 8 * st, ph) && wait_aside(bar_kv_empty + 8 * (kKS + st), ph);
                    if (!ok) break;
                    if (leader) {
                        const uint32_t full = bar_kv_full + 8 * st, dk = base + kOffK + st * kKVBytes, dv = base + kOffV + st * kKVBytes;
                        ptx::mbar_arrive_expect_tx(full, 2 * kKVBytes);
                        ptx::tma_load_4d(dk, &tm_k, full, 0, c[1], c[2], c[3]);
                        ptx::tma_load_4d(dk + kKVBytes / 2, &tm_k, full, 64, c[1], c[2], c[3]);
                        ptx::tma_load_4d(dv, &tm_v, full, 0, c[1], c[2], c[3]);
                        ptx::tma_load_4d(dv + kKVBytes / 2, &tm_v, full, 64, c[1], c[2], c[3]);
                    }
                }
            }
        } else {
            // ---------------- Q gather from the CTA's second tile on: the rows of one stream's tile after the other by TMA,
            // four rows of 64 columns per instruction, a lane four rows, as soon as a Q buffer is free.  The records are
            // read a stream ahead.  (128 rows take the TMA unit about 4600 cycles: hidden in the tile before.)
            ptx::prefetch_tensormap(&tm_q);
            const bool leader = ptx::elect_one();
            uint32_t k = 0, nq[2] = {1u, (ti.w & 0x1ff) > kHalf ? 1u : 0u};   // the epilogue warps gather the first tile's rows
            int n = blockIdx.x + gridDim.x, rows[4];   // the next tile: the second is the CTA's own as well
            auto fetch_rows = [&](const int4 &t, int xs) {   // a row beyond the tile's last one: that one again
                const int last = (t.w & 0x1ff) - 1;
#pragma unroll
                for (int u = 0; u < 4; ++u) rows[u] = p.recs[t.z + min(xs * kHalf + 4 * lane + u, last)].x;
            };
            // the next tile's entry, passed on to the other warps; the one after it is claimed
            auto next_tile = [&]() {
                if constexpr (kClaim) n = __shfl_sync(0xffffffffu, n, 0);
                const int4 t = n < n_tiles ? p.tiles[n] : make_int4(0, 0, 0, 0);
                ++k;
                if constexpr (kClaim) {
                    const int2 r = n < n_tiles ? p.ranges[n] : make_int2(0, 0);
                    if (lane == 0) n = atomicAdd(p.n_tiles + 2, 1) + 2 * gridDim.x;
                    if (!__all_sync(0xffffffffu, wait_aside(bar_t_empty + 8 * (k % kTS), ((k / kTS) & 1u) ^ 1u))) return make_int4(0, 0, 0, 0);
                    if (leader) {
                        meta->tile[k % kTS] = t;
                        meta->range[k % kTS] = r;
                        ptx::mbar_arrive(bar_t_full + 8 * (k % kTS));
                    }
                } else {
                    n += gridDim.x;
                }
                return t;
            };
            int4 next = ti;
            bool first = true, ok = true;
            while (ok && next.w) {
                ti = next;
                next = next_tile();
                if (first) {
                    first = false;
                    if (next.w) fetch_rows(next, 0);
                    continue;
                }
                const int bb = (unsigned)ti.x / (unsigned)p.Hkv, nx = kClaim && (ti.w & 0x1ff) > kHalf ? 2 : 1;   // (dealt: the epilogue warps take the second stream's)
#pragma unroll 1
                for (int x = 0; x < nx; ++x) {
                    const uint32_t turn = x ? nq[1]++ : nq[0]++, qs = 2 * (turn & 1u) + x, full = bar_q_full + 8 * qs;
                    ok = __all_sync(0xffffffffu, wait_aside(bar_q_empty + 8 * qs, ((turn >> 1) & 1u) ^ 1u));
                    if (!ok) break;
                    if (leader) {
                        ptx::mbar_arrive_expect_tx(full, kQBytes);
                        ptx::mbar_arrive(full);
                        ptx::mbar_arrive(full);
                        ptx::mbar_arrive(full);
                    }
                    int at[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) at[u] = q_row(rows[u], bb);
                    __syncwarp();
                    const uint32_t dst = base + kOffQ + qs * kQBytes + lane * 512;
                    ptx::tma_gather4(dst, &tm_q, full, 0, at[0], at[1], at[2], at[3]);
                    ptx::tma_gather4(dst + kQBytes / 2, &tm_q, full, 64, at[0], at[1], at[2], at[3]);
                    const bool more = x + 1 < nx;
                    const int4 t = more ? ti : next;
                    if (t.w) fetch_rows(t, more);
                }
            }
        }
    } else if (warp >= 8) {
        // ---------------- epilogue warps: normalised piece outputs and their log-sum-exps, one thread per row
        ptx::setmaxnreg_dec<kRegsEpi>();
        const int row = tid & 127;
        const uint32_t lane_addr = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        uint32_t k = 0;
        bool ok = true;
        warp_read(0);
        // Q rows of a stream's tile by 16-byte copies, two rows (16 lanes each) per instruction
        auto copy_rows = [&](const int4 &t, int x, uint32_t buf) {
            const int cnt = t.w & 0x1ff, chunk = lane & 15, odd = lane >> 4, bb = (unsigned)t.x / (unsigned)p.Hkv;
            const uint32_t dst = base + kOffQ + buf * kQBytes + (chunk >> 3) * (kQBytes / 2) + ((warp & 3) * 32 + odd) * 128;
            const int at = q_row(p.recs[t.z + min(x * kHalf + row, cnt - 1)].x, bb);
#pragma unroll 4
            for (int i = 0; i < 16; ++i) {
                const int from = __shfl_sync(0xffffffffu, at, 2 * i + odd);
                ptx::cp_async16(dst + i * 256 + (((chunk & 7) ^ ((2 * i + odd) & 7)) << 4), p.q + from * p.q_pitch + chunk * 8);
            }
        };
        auto rows_copied = [&](uint32_t buf) {   // (no barrier among the four warps: one whose wait ran out would leave them there)
            ptx::cp_async_wait_all();
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar_q_full + 8 * buf);
        };
        // the CTA's first tile
#pragma unroll 1
        for (int x = 0; x * kHalf < (ti.w & 0x1ff); ++x) {
            copy_rows(ti, x, x);
            rows_copied(x);
        }
        // Where the tiles are dealt their walks may be shorter than the gather of their rows by TMA (4600 cycles a stream): the
        // second stream's rows are copied here, two tiles ahead, behind the tile whose buffer they take, and handed over before
        // the next one's results.  1999 positions, 32/8 heads, four spans (walks of two to three blocks): kernel 47.3 -> 41.5 us.
        uint32_t nq = (ti.w & 0x1ff) > kHalf ? 1u : 0u;
        int copied = -1;   // buffer
        auto copy_ahead = [&](int n) {
            const int4 t = n < n_tiles ? p.tiles[n] : make_int4(0, 0, 0, 0);
            if ((t.w & 0x1ff) > kHalf) {
                copied = 2 * (nq & 1u) + 1;
                const bool got = __all_sync(0xffffffffu, wait_aside(bar_q_empty + 8 * copied, ((nq >> 1) & 1u) ^ 1u));
                ++nq;
                if (!got) return false;
                copy_rows(t, 1, copied);
            }
            return true;
        };
        if constexpr (!kClaim) ok = copy_ahead(blockIdx.x + gridDim.x);
        uint32_t tx[2] = {0, 0};
        while (ok && ti.w) {
            const int cnt = ti.w & 0x1ff, nx = cnt > kHalf ? 2 : 1, rec0 = ti.z;
            ok = take_tile(++k);
            if constexpr (!kClaim) {
                if (copied >= 0) rows_copied(copied);
                copied = -1;
            }
#pragma unroll 1
            for (int x = 0; x < nx && ok; ++x) {
                const uint32_t t = x ? tx[1] : tx[0];
                const int r = x * kHalf + row;
                const bool valid = r < cnt;
                const int2 rs = valid ? *reinterpret_cast<const int2 *>(&p.recs[rec0 + r]) : make_int2(0, 0);
                const long long slot = (long long)rs.x * p.slots + rs.y;
                __half *dst = p.part_o + slot * kD;
                ok = __all_sync(0xffffffffu, wait_aside(bar_l_full + 8 * x, t & 1u) && wait_aside(bar_o_full + 8 * x, t & 1u));
                if (!ok) break;
                ptx::tc_fence_after();
                const float2 stat = meta->stats[r];
                uint32_t exps = 0;   // biased exponent of each 32-column chunk's largest magnitude
                // one 32-column chunk: block exponent, fp16 mantissas, two 32-byte stores
#pragma unroll 1
                for (int q4 = 0; q4 < 4; ++q4) {
                    uint32_t o[32];
                    ptx::tmem_ld32(lane_addr + kColO + x * kD + q4 * 32, o);
                    ptx::tmem_wait_ld();
                    if (q4 == 3) {
                        // O is in registers: the next tile's first PV may overwrite it
                        ptx::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(bar_o_empty + 8 * x);
                    }
                    if (valid) {
                        float am[2] = {0.f, 0.f};
#pragma unroll
                        for (int cc = 0; cc < 32; cc += 4)
#pragma unroll
                            for (int u = 0; u < 2; ++u)
                                am[u] = max3(am[u], fabsf(__uint_as_float(o[cc + 2 * u])), fabsf(__uint_as_float(o[cc + 2 * u + 1])));
                        const float amax = fmaxf(am[0], am[1]) * stat.x;
                        uint32_t eb = (__float_as_uint(amax) >> 23) & 0xffu;
                        eb = eb < 1u ? 1u : (eb > 252u ? 252u : eb);
                        exps |= eb << (8 * q4);
                        // normalisation and 2^(126 - eb), which brings the chunk into [-1, 1], in one factor
                        const float down = stat.x * __uint_as_float((253u - eb) << 23);
#pragma unroll
                        for (int s8 = 0; s8 < 2; ++s8) {
                            uint32_t w[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const __half2 pp = __floats2half2_rn(__uint_as_float(o[s8 * 16 + 2 * e]) * down,
                                                                     __uint_as_float(o[s8 * 16 + 2 * e + 1]) * down);
                                w[e] = *reinterpret_cast<const uint32_t *>(&pp);
                            }
                            ptx::st_global_v8(dst + q4 * 32 + s8 * 16, w);
                        }
                    }
                }
                if (valid) p.part_lse[slot] = make_float2(stat.y, __uint_as_float(exps));
                if (x) ++tx[1]; else ++tx[0];
            }
            if constexpr (!kClaim) {
                if (ok) ok = copy_ahead(blockIdx.x + (k + 1) * gridDim.x);
            }
        }
    } else {
        // ---------------- row warps of stream x: softmax per 64-key block, one thread per row
        ptx::setmaxnreg_inc<kRegsRow>();
        const int x = warp >> 2, row = tid & 127, r = x * kHalf + row;
        const uint32_t lane_addr = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t o_addr = lane_addr + kColO + x * kD, s_col = lane_addr + kColS + x * (2 * kBK);
        auto interval = [&](const int4 &t) {   // {lo, hi} of this thread's piece
            return r < (t.w & 0x1ff) ? *reinterpret_cast<const int2 *>(&p.recs[t.z + r].z) : make_int2(INT_MAX, -1);
        };
        uint32_t n = 0, na = 0, t = 0;   // blocks and tiles of the stream so far; all blocks of the CTA
        uint32_t k = 0;
        bool ok = true;
        rg = first_range();
        warp_read(0);
        int2 iv = interval(ti);
        while (ok && ti.w) {
            const int nblk = ti.w >> 9, range = x ? rg.y : rg.x, first_block = range & 0xffff, end_block = range >> 16;
            int k0 = (ti.y + 1 - nblk + first_block) * kBK;
            ok = take_tile(++k);
            if (!ok) break;
            const int2 iv_next = interval(ti);   // requested a tile ahead
            if (first_block < end_block) {
                const int lo = iv.x, hi = iv.y;
                float m_ref = -CUDART_INF_F, l = 0.f;
#pragma unroll 1
                for (int j = first_block; j < end_block; ++j, ++n, k0 += kBK) {
                    const uint32_t b = n & 1u, ph = (n >> 1) & 1u;
                    ok = ptx::mbar_wait_warp(bar_s_full + 16 * x + 8 * b, ph, abort_flag);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    uint32_t sr[2][32];
                    ptx::tmem_ld32(s_col + b * kBK, sr[0]);
                    ptx::tmem_ld32(s_col + b * kBK + 32, sr[1]);
                    ptx::tmem_wait_ld();
                    const bool any = k0 <= hi && k0 + kBK - 1 >= lo;
                    if (!(any && k0 >= lo && k0 + kBK - 1 <= hi)) {
                        // bit c of the mask: column c of the block lies inside the piece
                        const int ca = lo > k0 ? lo - k0 : 0, cb = hi - k0 < kBK - 1 ? hi - k0 : kBK - 1;
                        const unsigned long long inside = any ? (~0ull >> (63 - (cb - ca))) << ca : 0ull;
                        const uint32_t in2[2] = {static_cast<uint32_t>(inside), static_cast<uint32_t>(inside >> 32)};
#pragma unroll
                        for (int hlf = 0; hlf < 2; ++hlf)
#pragma unroll
                            for (int cc = 0; cc < 32; ++cc)
                                if (!(in2[hlf] & (1u << cc))) sr[hlf][cc] = 0xff800000u;   // -inf
                    }
                    // block maximum on the raw logits (softmax_scale > 0 on this path), four independent chains
                    float bm;
                    {
                        float mx[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
                        for (int hlf = 0; hlf < 2; ++hlf)
#pragma unroll
                            for (int cc = 0; cc < 32; cc += 8)
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    mx[u] = max3(mx[u], __uint_as_float(sr[hlf][cc + 2 * u]), __uint_as_float(sr[hlf][cc + 2 * u + 1]));
                        bm = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * p.scale2;
                    }
                    // running reference maximum; O is rescaled only when it moves by more than the threshold
                    const bool first = (l == 0.f);   // no key of this row seen so far
                    const bool need = !first && (bm > m_ref + kRescaleThreshold);
                    if (__any_sync(0xffffffffu, need)) {
                        // PV of the block before must have landed before O is touched
                        const uint32_t np = na + j - 1u;
                        ok = ptx::mbar_wait_warp(bar_kv_empty + 8 * (x * kKS + np % kKS), (np / kKS) & 1u, abort_flag);
                        if (!ok) break;
                        ptx::tc_fence_after();
                        const float f = need ? ex2_approx(m_ref - bm) : 1.f;
#pragma unroll 1
                        for (int q8 = 0; q8 < 8; ++q8) {
                            uint32_t o[16];
                            ptx::tmem_ld16(o_addr + q8 * 16, o);
                            ptx::tmem_wait_ld();
#pragma unroll
                            for (int cc = 0; cc < 16; ++cc) o[cc] = __float_as_uint(__uint_as_float(o[cc]) * f);
                            ptx::tmem_st16(o_addr + q8 * 16, o);
                        }
                        if (need) { l *= f; m_ref = bm; }
                    }
                    if (first && bm > -CUDART_INF_F) m_ref = bm;   // first keys of this row
                    uint32_t pk[32];
                    {
                        // p = 2^(s*scale - m_ref), two columns per packed fp32x2 instruction; masked columns
                        // hold -inf and give 0 (a row with no key so far has m_ref = -inf: it subtracts 0)
                        const float neg_m = m_ref > -CUDART_INF_F ? -m_ref : 0.f;
                        const unsigned long long sc2 = pack2(p.scale2, p.scale2), nm2 = pack2(neg_m, neg_m);
                        unsigned long long acc2[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) acc2[u] = pack2(0.f, 0.f);
#pragma unroll
                        for (int cc = 0; cc < 32; ++cc) {
                            const int hlf = cc >> 4, c2 = (cc & 15) * 2;
                            const unsigned long long y = ffma2(
                                pack2(__uint_as_float(sr[hlf][c2]), __uint_as_float(sr[hlf][c2 + 1])), sc2, nm2);
                            float y0, y1;
                            unpack2(y, y0, y1);
                            const float p0 = ex2_approx(y0), p1 = ex2_approx(y1);
                            acc2[cc & 3] = fadd2(acc2[cc & 3], pack2(p0, p1));
                            const __nv_bfloat162 pp = __floats2bfloat162_rn(p0, p1);
                            pk[cc] = *reinterpret_cast<const uint32_t *>(&pp);
                        }
                        float s0, s1, s2, s3;
                        unpack2(fadd2(acc2[0], acc2[1]), s0, s1);
                        unpack2(fadd2(acc2[2], acc2[3]), s2, s3);
                        l += (s0 + s1) + (s2 + s3);
                    }
                    ptx::tmem_st32(s_col + b * kBK, pk);
                    ptx::tmem_wait_st();
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar_p_ready + 16 * x + 8 * b);
                }
                // the epilogue has read the statistics (and O) of the tile before
                if (ok && t > 0) ok = ptx::mbar_wait_warp(bar_o_empty + 8 * x, (t - 1u) & 1u, abort_flag);
                ++t;
                if (ok) {
                    meta->stats[r] = make_float2(l > 0.f ? 1.f / l : 0.f, l > 0.f ? m_ref + log2f(l) : -CUDART_INF_F);
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar_l_full + 8 * x);
                }
            }
            na += nblk;
            iv = iv_next;
        }
    }

    // ---- teardown
    __syncthreads();
    if (*abort_flag) {
        if (tid == 0) atomicOr(p.status, kStatusTimeout);
        __nanosleep(200000);   // let copies and MMAs that may still be in flight land
        __syncthreads();
    }
    if (warp == 12) {
        __syncwarp();
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------
// The rows of Q of a chunk as a dense [B, Hq, Lc, 128] tensor, where its strides have no common row pitch.  16 threads per
// row.  Bound by HBM.  The attention call with the tokens of 32 heads 4104 elements apart, four spans: 512
// positions 42 us, 16384 606 us (with a strided copy per head 136 and 958 us; dense queries 38 and 563 us).
__global__ void __launch_bounds__(256)
copy_q_rows(const bf16 *__restrict__ q, Call c, long long r0, int Lc, bf16 *__restrict__ dst) {
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x, row = gid >> 4;
    chain_wait();
    chain_release();
    if (row >= (long long)c.B * c.Hq * Lc) return;
    const int sub = (int)(gid & 15), bh = (int)((unsigned)row / (unsigned)Lc), rc = (int)((unsigned)row % (unsigned)Lc);   // rows < 2^31
    const bf16 *src = q + (bh / c.Hq) * c.q_sb + (bh % c.Hq) * c.q_sh + (r0 + rc) * c.q_st + sub * 8;
    *reinterpret_cast<uint4 *>(dst + row * kD + sub * 8) = __ldg(reinterpret_cast<const uint4 *>(src));
}

// dst += w x (eight columns of a piece's block-floating-point output; `exps` holds the chunk exponents)
__device__ __forceinline__ void add_piece(const uint4 &raw, float exps, int sub, float w, float (&dst)[8]) {
    const uint32_t eb = (__float_as_uint(exps) >> (8 * (sub >> 2))) & 0xffu;
    const float ws = w * __uint_as_float((eb + 1u) << 23);   // weight x 2^(eb - 126)
    const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&rw[e]));
        dst[2 * e] = fmaf(ws, f.x, dst[2 * e]);
        dst[2 * e + 1] = fmaf(ws, f.y, dst[2 * e + 1]);
    }
}

// Per row: merge the normalised piece outputs through their log-sum-exp, for few rows or many slots.  16 lanes per row, 8 columns
// each; every lane works out the row's weights.
// Bound by a row's chain of loads, which tc_merge below makes longer.  Few rows, this and tc_merge (ncu): 100, 150 and 300 positions, 32 heads,
// eight spans 4.5, 4.5 and 6.0 us, 5.2, 5.2 and 7.8; 500 positions 6.8 and 7.0, 1000 11.3 and 11.1.  Many slots, this and tc_merge with four and with two
// rows a warp: 64 spans over 16384 keys, 600, 1200, 1800 and 4500 positions 34, 61, 85 and 199 us, 36, 63, 91 and 208, 33, 59, 82 and 201; from the
// start, a piece or two in most rows, 1800 and 4500 positions 14 and 33 us, 14 and 32, 22 and 52.  With 32 spans four rows a warp are
// ahead where rows have many pieces: 1000, 1400 and 4500 positions 40, 52 and 145 us, 36, 49 and 138.
__global__ void __launch_bounds__(256)
tc_merge_few(const __half *__restrict__ part_o, const float2 *__restrict__ part_lse,
             const unsigned char *__restrict__ n_pieces, Call c, int slots, int Lc, long long r0,
             bf16 *__restrict__ out, float *__restrict__ lse) {
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long row = gid >> 4;
    const int sub = (int)(gid & 15);
    const long long rows = (long long)c.B * c.Hq * Lc;
    chain_wait();
    if (row >= rows) return;
    const int cnt = n_pieces[row];
    const float2 *pl = part_lse + row * slots;
    const __half *po = part_o + row * slots * kD + sub * 8;
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    // running maximum and denominator (log2 domain); the pieces come four at a time so that their loads are in flight together
    float mx = -CUDART_INF_F, den = 0.f;
    for (int j0 = 0; j0 < cnt; j0 += 4) {
        float2 pj[4];
        uint4 raw[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool on = j0 + u < cnt;
            pj[u] = on ? __ldg(pl + j0 + u) : make_float2(-CUDART_INF_F, 0.f);
            raw[u] = on ? __ldg(reinterpret_cast<const uint4 *>(po + (long long)(j0 + u) * kD)) : make_uint4(0, 0, 0, 0);
        }
        const float bm = fmaxf(fmaxf(pj[0].x, pj[1].x), fmaxf(pj[2].x, pj[3].x));
        if (bm > mx) {
            const float r = mx == -CUDART_INF_F ? 0.f : exp2f(mx - bm);
            den *= r;
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] *= r;
            mx = bm;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (pj[u].x == -CUDART_INF_F) continue;
            const float w = exp2f(pj[u].x - mx);
            den += w;
            add_piece(raw[u], pj[u].y, sub, w, acc);
        }
    }
    const float inv = den > 0.f ? 1.f / den : 0.f;
    const int rc = (int)((unsigned)row % (unsigned)Lc);   // rows < 2^31
    const int bh = (int)((unsigned)row / (unsigned)Lc);
    const int h = bh % c.Hq, b = bh / c.Hq;
    const long long r = r0 + rc;
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 pp = __floats2bfloat162_rn(acc[2 * e] * inv, acc[2 * e + 1] * inv);
        w[e] = *reinterpret_cast<const uint32_t *>(&pp);
    }
    *reinterpret_cast<uint4 *>(out + b * c.q_sb + h * c.q_sh + r * c.q_st + sub * 8) = make_uint4(w[0], w[1], w[2], w[3]);
    if (sub == 0)
        lse[((long long)b * c.Hq + h) * c.Lq + r] = den > 0.f ? (mx + log2f(den)) * kLn2 : -CUDART_INF_F;
}

// Per row: merge the normalised piece outputs through their log-sum-exp.  A warp takes per_warp consecutive rows (a power of
// two, kMergeLeast to 32): first 32 / per_warp lanes each work out a row's weights and write its lse, then every half of the warp adds up
// every other row's pieces, 8 columns per lane, four pieces at a time with the next four already requested.  The last rows come
// first: their partial results were written last, and what the L2 still holds of them is read from there.
// Bound by the reads of the partial results (3.2 GB at 65536 positions, 32 heads, eight spans: 6.6 TB/s).  With 16 lanes that
// all worked out their row's weights, issue slots were 72 % used and the loads of a row waited for the sum of the one before:
// 637 us, and 480 like this; 16384 positions 152 and 114 us, 1999 positions, four spans 19.6 and 15.7 (ncu).
// Rows of a warp: up to kMergePieces slots -- fewer pieces in a row cost more for the weights, more make the last warps' turn
// long -- and as many warps as keep the loads going.  16 and 8 rows of 16 slots: 131072 rows 101 and 97 us (93 before); 32 and 16 rows of 2
// slots: 960000 rows 123 and 129 us (207 before); 16, 8 and 4 rows of 8 slots: 128000 rows 40, 44 and 46 us (47 before), 16000 rows
// 16.0, 12.0 and 10.4 (10.2 before).
constexpr int kMergeWarps = 4;      // of a CTA
constexpr int kMergePieces = 128;   // slots a warp takes at most
constexpr int kMergeFill = 19;      // warps an SM at least
constexpr int kMergeLeast = 4;      // rows a warp takes at least; where the two above allow fewer: tc_merge_few
__global__ void __launch_bounds__(kMergeWarps * 32, 8)
tc_merge(const __half *__restrict__ part_o, const float2 *__restrict__ part_lse,
         const unsigned char *__restrict__ n_pieces, Call c, int slots, int Lc, long long r0, int per_warp,
         bf16 *__restrict__ out, float *__restrict__ lse) {
    extern __shared__ float2 s_weight[];   // [rows of the CTA][slots, an odd number] {weight, chunk exponents; 0: no part in the result}
    const int lane = threadIdx.x & 31;
    const long long row0 = ((long long)(gridDim.x - 1 - blockIdx.x) * kMergeWarps + (threadIdx.x >> 5)) * per_warp;
    const long long rows = (long long)c.B * c.Hq * Lc;
    chain_wait();
    if (row0 >= rows) return;
    // ---- weights: 32 / per_warp lanes per row
    const int lanes = 32 / per_warp, pitch = slots | 1;   // odd: the lanes' rows start in different banks
    __shared__ int4 s_row[kMergeWarps][32];   // {offset of the row in `out` (two words), reciprocal denominator, pieces}
    int4 *rows_of = s_row[threadIdx.x >> 5];
    float2 *sw = s_weight + (threadIdx.x >> 5) * per_warp * pitch;
    {
        const int own = lane / lanes, first = lane % lanes;
        const long long row = row0 + own < rows ? row0 + own : rows - 1;   // rows past the last: that one again
        const int cnt = n_pieces[row];
        const float2 *pl = part_lse + row * slots;
        float2 *mine = sw + own * pitch;
        float mx = -CUDART_INF_F, den = 0.f;
#pragma unroll 4
        for (int j = first; j < cnt; j += lanes) {
            const float2 pj = __ldg(pl + j);
            mine[j] = pj;
            mx = fmaxf(mx, pj.x);
        }
        for (int o = 1; o < lanes; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        for (int j = first; j < cnt; j += lanes) {
            const float2 pj = mine[j];
            const bool on = pj.x != -CUDART_INF_F;
            const float w = on ? exp2f(pj.x - mx) : 0.f;
            den += w;
            mine[j] = make_float2(w, on ? pj.y : 0.f);
        }
        for (int o = 1; o < lanes; o <<= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
        const int rc = (int)((unsigned)row % (unsigned)Lc);   // rows < 2^31
        const int bh = (int)((unsigned)row / (unsigned)Lc);
        const int h = bh % c.Hq, b = bh / c.Hq;
        const long long r = r0 + rc, off = b * c.q_sb + h * c.q_sh + r * c.q_st;
        if (first == 0) {
            rows_of[own] = make_int4((int)off, (int)(off >> 32), __float_as_int(den > 0.f ? 1.f / den : 0.f), cnt);
            lse[((long long)b * c.Hq + h) * c.Lq + r] = den > 0.f ? (mx + log2f(den)) * kLn2 : -CUDART_INF_F;
        }
    }
    __syncwarp();
    // ---- 16 lanes per row: its pieces four at a time, the next four (of this row or of the next but one) requested before the
    // ones in hand are added up
    const int sub = lane & 15, shift = 8 * (sub >> 2);
    const int last = (int)(rows - 1 - row0 < per_warp - 1 ? rows - 1 - row0 : per_warp - 1);
    const __half *po = part_o + row0 * slots * kD + sub * 8;
    auto load = [&](uint4 (&raw)[4], int row, int j, int n) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (j + u < n) raw[u] = __ldg(reinterpret_cast<const uint4 *>(po + (long long)(row * slots + j + u) * kD));
    };
    unsigned long long acc[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[e] = pack2(0.f, 0.f);
    auto add = [&](const uint4 (&raw)[4], int row, int j, int n) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j + u >= n) break;
            const float2 w = sw[row * pitch + j + u];
            const uint32_t exps = __float_as_uint(w.y);
            if (exps == 0u) continue;
            const float ws = w.x * __uint_as_float((((exps >> shift) & 0xffu) + 1u) << 23);   // weight x 2^(eb - 126)
            const unsigned long long ww = pack2(ws, ws);
            const uint32_t rw[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&rw[e]));
                acc[e] = ffma2(pack2(f.x, f.y), ww, acc[e]);
            }
        }
    };
    int row = lane >> 4, j = 0, n = row <= last ? rows_of[row].w : 0;
    uint4 raw[2][4];
    load(raw[0], row, j, n);
    for (;;) {
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            int row2 = row, j2 = j + 4, n2 = n;
            if (j2 >= n) {
                row2 = row + 2;
                j2 = 0;
                n2 = row2 <= last ? rows_of[row2].w : 0;
            }
            load(raw[y ^ 1], row2, j2, n2);
            add(raw[y], row, j, n);
            if (row2 != row) {
                if (row <= last) {
                    const int4 ri = rows_of[row];
                    const float f = __int_as_float(ri.z);
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float a0, a1;
                        unpack2(acc[e], a0, a1);
                        const __nv_bfloat162 pp = __floats2bfloat162_rn(a0 * f, a1 * f);
                        w[e] = *reinterpret_cast<const uint32_t *>(&pp);
                        acc[e] = pack2(0.f, 0.f);
                    }
                    const long long off = (long long)(((unsigned long long)(unsigned)ri.y << 32) | (unsigned)ri.x);
                    *reinterpret_cast<uint4 *>(out + off + sub * 8) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            row = row2; j = j2; n = n2;
        }
        if (!__any_sync(0xffffffffu, row <= last)) break;
    }
}

// Per row, per-span mode (Algorithm 1 with the gate of Section "Combination"): slot j holds the
// attention over the part of S_t left of the window, slot top_k the attention over the window; A_t
// merges the two through their log-sum-exp, and O = sum_t alpha_t A_t with alpha = softmax of the
// selected anchors' search scores.  16 threads per row, 8 columns each.
__global__ void __launch_bounds__(256)
tc_merge_gated(const __half *__restrict__ part_o, const float2 *__restrict__ part_lse,
               const int32_t *__restrict__ anchor, const float *__restrict__ score, Call c, int slots, int Lc,
               long long r0, bf16 *__restrict__ out, float *__restrict__ lse, float *__restrict__ lse_span) {
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long row = gid >> 4;
    const int sub = (int)(gid & 15);
    const long long rows = (long long)c.B * c.Hq * Lc;
    chain_wait();
    if (row >= rows) return;
    const int rc = (int)((unsigned)row % (unsigned)Lc);   // rows < 2^31
    const int bh = (int)((unsigned)row / (unsigned)Lc);
    const int h = bh % c.Hq, b = bh / c.Hq;
    const long long r = r0 + rc, i = c.q_pos0 + r;
    const long long orow = ((long long)b * c.Hq + h) * c.Lq + r;
    const int32_t *an = anchor + orow * c.top_k;
    const float *sc = score + orow * c.top_k;
    const float2 *pl = part_lse + row * slots;
    const long long ell = base_len(c, i);
    const long long w_lo = i - c.window + 1 > 0 ? i - c.window + 1 : 0;
    const bool has_w = c.window > 0;
    // the window piece is needed by nearly every row: request it with the first loads
    const float2 pw = has_w ? __ldg(pl + c.top_k) : make_float2(-CUDART_INF_F, 0.f);
    const uint4 raw_w = has_w ? __ldg(reinterpret_cast<const uint4 *>(part_o + (row * slots + c.top_k) * kD + sub * 8))
                              : make_uint4(0, 0, 0, 0);
    const float lw = pw.x;

    float smax = -CUDART_INF_F;
    int n_sel = 0;
    for (int j = 0; j < c.top_k; ++j)
        if (an[j] >= 0 && an[j] <= i) { smax = fmaxf(smax, sc[j]); ++n_sel; }
    float sden = 0.f;
    for (int j = 0; j < c.top_k; ++j)
        if (an[j] >= 0 && an[j] <= i) sden += expf(sc[j] - smax);
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    // O = sum_t alpha_t (w_t o_t + ww_t o_W) / den_t: the window piece enters once, with the summed
    // coefficient cw; the spans' pieces come four at a time so that their loads are in flight together
    float lse_first = -CUDART_INF_F, cw = 0.f;
    if (n_sel == 0 && has_w) {   // Algorithm 1, empty selection: the window alone
        cw = 1.f;
        lse_first = lw * kLn2;
    }
    bool first = true;
    const __half *po = part_o + row * slots * kD + sub * 8;
    for (int j0 = 0; j0 < c.top_k; j0 += 4) {
        float2 pj[4];
        uint4 raw[4];
        bool sel[4], has_s[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u;
            const long long t = j < c.top_k ? an[j] : -1;
            sel[u] = t >= 0 && t <= i;
            const long long a = t - (long long)c.back * ell;
            has_s[u] = sel[u] && (!has_w || (a > 0 ? a : 0) < w_lo);   // a part of S_t lies left of the window
            pj[u] = has_s[u] ? __ldg(pl + j) : make_float2(-CUDART_INF_F, 0.f);
            raw[u] = has_s[u] ? __ldg(reinterpret_cast<const uint4 *>(po + (long long)j * kD)) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u;
            if (j >= c.top_k) break;
            float l_t = -CUDART_INF_F;
            if (sel[u]) {
                const float lj = pj[u].x;
                const float m = fmaxf(lj, lw);
                const float wj = has_s[u] ? exp2f(lj - m) : 0.f, ww = has_w ? exp2f(lw - m) : 0.f;
                const float den = wj + ww;
                const float alpha = expf(sc[j] - smax) / sden;
                cw = fmaf(alpha, ww / den, cw);
                if (has_s[u]) {
                    const uint32_t eb = (__float_as_uint(pj[u].y) >> (8 * (sub >> 2))) & 0xffu;
                    const float ws = alpha * wj / den * __uint_as_float((eb + 1u) << 23);   // weight x 2^(eb - 126)
                    const uint32_t rw[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&rw[e]));
                        acc[2 * e] = fmaf(ws, f.x, acc[2 * e]);
                        acc[2 * e + 1] = fmaf(ws, f.y, acc[2 * e + 1]);
                    }
                }
                l_t = (m + log2f(den)) * kLn2;
                if (first) { lse_first = l_t; first = false; }
            }
            if (lse_span && sub == 0) lse_span[orow * c.top_k + j] = l_t;
        }
    }
    if (cw != 0.f) add_piece(raw_w, pw.y, sub, cw, acc);
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 pp = __floats2bfloat162_rn(acc[2 * e], acc[2 * e + 1]);
        w[e] = *reinterpret_cast<const uint32_t *>(&pp);
    }
    *reinterpret_cast<uint4 *>(out + b * c.q_sb + h * c.q_sh + r * c.q_st + sub * 8) = make_uint4(w[0], w[1], w[2], w[3]);
    if (sub == 0) lse[orow] = lse_first;
}

// The same for top_k <= K, K at most 8, arranged so that the per-row arithmetic (gate, log-sum-exp weights, base
// span length) is done once per row: a warp takes 32 consecutive rows; first every lane works out the
// coefficients of its own row (weight of every span piece, summed weight of the window piece, the
// log-sum-exps), then the warp walks its rows two at a time, 16 lanes per row and 8 columns per lane,
// with the coefficients handed over by shuffles.
// Bound by the reads of the partial results: with room for eight spans whatever top_k is, 106 registers and the shuffles of
// absent spans made it 402 us for 32768 positions, 32 heads, two spans and a window (1.1 GB, 2.7 TB/s); with room for two,
// 48 registers and 213 us; with the next two rows' pieces requested ahead 64 registers and 170 us (6.4 TB/s).  Eight spans 993 and 581 us,
// five 723 and 493, but four 265 and 281 (122 registers, two CTAs an SM): built for four it requests them in the same step, 270 us with 72
// registers.  (With 64, four CTAs an SM, 255 us, but search to merge of 500 positions at 16384, three and four spans, takes 138 and 154 us
// instead of 127 and 144.)
constexpr int kGateK = 8;
template <int K>
__global__ void __launch_bounds__(256, K <= 2 ? 4 : 1)
tc_merge_gated_rows(const __half *__restrict__ part_o, const float2 *__restrict__ part_lse,
                    const int32_t *__restrict__ anchor, const float *__restrict__ score, Call c, int slots, int Lc,
                    long long r0, bf16 *__restrict__ out, float *__restrict__ lse, float *__restrict__ lse_span) {
    const int lane = threadIdx.x & 31;
    const long long row0 = ((long long)(gridDim.x - 1 - blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32;
    const long long rows = (long long)c.B * c.Hq * Lc;
    chain_wait();
    if (row0 >= rows) return;
    const bool has_w = c.window > 0;
    // ---- phase A: lane = row
    float coef[K], cw = 0.f;       // weights of the span pieces and of the window piece
    uint32_t ex[K], ex_w = 0u;     // their chunk exponents
    long long out_off = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) { coef[j] = 0.f; ex[j] = 0u; }
    {
        const long long row = row0 + lane;
        if (row < rows) {
            const int rc = (int)((unsigned)row % (unsigned)Lc);   // rows < 2^31
            const int bh = (int)((unsigned)row / (unsigned)Lc);
            const int h = bh % c.Hq, b = bh / c.Hq;
            const long long r = r0 + rc, i = c.q_pos0 + r;
            const long long orow = ((long long)b * c.Hq + h) * c.Lq + r;
            out_off = b * c.q_sb + h * c.q_sh + r * c.q_st;
            const int32_t *an = anchor + orow * c.top_k;
            const float *sc = score + orow * c.top_k;
            const float2 *pl = part_lse + row * slots;
            const long long ell = base_len(c, i);
            const long long w_lo = i - c.window + 1 > 0 ? i - c.window + 1 : 0;
            const float2 pw = has_w ? __ldg(pl + c.top_k) : make_float2(-CUDART_INF_F, 0.f);
            const float lw = pw.x;
            ex_w = __float_as_uint(pw.y);
            float scv[K], lj[K];
            bool sel[K], has_s[K];
            float smax = -CUDART_INF_F;
            int n_sel = 0;
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const long long t = j < c.top_k ? an[j] : -1;
                sel[j] = t >= 0 && t <= i;
                scv[j] = sel[j] ? sc[j] : -CUDART_INF_F;
                const long long a = t - (long long)c.back * ell;
                has_s[j] = sel[j] && (!has_w || (a > 0 ? a : 0) < w_lo);   // a part of S_t lies left of the window
                const float2 pj = has_s[j] ? __ldg(pl + j) : make_float2(-CUDART_INF_F, 0.f);
                lj[j] = pj.x;
                ex[j] = __float_as_uint(pj.y);
                if (sel[j]) { smax = fmaxf(smax, scv[j]); ++n_sel; }
            }
            float sden = 0.f;
#pragma unroll
            for (int j = 0; j < K; ++j)
                if (sel[j]) sden += expf(scv[j] - smax);
            float lse_first = -CUDART_INF_F;
            if (n_sel == 0 && has_w) {   // Algorithm 1, empty selection: the window alone
                cw = 1.f;
                lse_first = lw * kLn2;
            }
            bool first = true;
#pragma unroll
            for (int j = 0; j < K; ++j) {
                if (j >= c.top_k) break;
                float l_t = -CUDART_INF_F;
                if (sel[j]) {
                    const float m = fmaxf(lj[j], lw);
                    const float wj = has_s[j] ? exp2f(lj[j] - m) : 0.f, ww = has_w ? exp2f(lw - m) : 0.f;
                    const float den = wj + ww;
                    const float alpha = expf(scv[j] - smax) / sden;
                    cw = fmaf(alpha, ww / den, cw);
                    coef[j] = has_s[j] ? alpha * wj / den : 0.f;
                    l_t = (m + log2f(den)) * kLn2;
                    if (first) { lse_first = l_t; first = false; }
                }
                if (lse_span) lse_span[orow * c.top_k + j] = l_t;
            }
            lse[orow] = lse_first;
        }
    }
    // ---- phase B: two rows per step, 16 lanes per row
    const int sub = lane & 15, hi = lane >> 4;
    const int shift = 8 * (sub >> 2);
    constexpr bool kAhead = K != 4;   // a step's pieces are requested before the sums of the one before
    float cf[2][K + 1];
    uint32_t ee[2][K + 1];
    uint4 raw[2][K + 1];
    auto fetch = [&](int rr, float (&cf)[K + 1], uint32_t (&ee)[K + 1], uint4 (&raw)[K + 1]) {
        const int src = 2 * rr + hi;
        const __half *po = part_o + (row0 + src) * slots * kD + sub * 8;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            cf[j] = __shfl_sync(0xffffffffu, coef[j], src);
            ee[j] = __shfl_sync(0xffffffffu, ex[j], src);
        }
        cf[K] = __shfl_sync(0xffffffffu, cw, src);
        ee[K] = __shfl_sync(0xffffffffu, ex_w, src);
#pragma unroll
        for (int j = 0; j <= K; ++j)
            if (cf[j] != 0.f) raw[j] = __ldg(reinterpret_cast<const uint4 *>(po + (long long)(j < K ? j : c.top_k) * kD));
    };
    if constexpr (kAhead) fetch(0, cf[0], ee[0], raw[0]);
#pragma unroll (kAhead ? 2 : 4)
    for (int rr = 0; rr < 16; ++rr) {
        const int now = kAhead ? rr & 1 : 0;
        const int src = 2 * rr + hi;
        const long long row = row0 + src;
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.f;
        const long long off = __shfl_sync(0xffffffffu, out_off, src);
        if constexpr (kAhead) {
            if (rr + 1 < 16) fetch(rr + 1, cf[now ^ 1], ee[now ^ 1], raw[now ^ 1]);
        } else {
            fetch(rr, cf[0], ee[0], raw[0]);
        }
#pragma unroll
        for (int j = 0; j <= K; ++j)
            if (cf[now][j] != 0.f) {
                const uint32_t eb = (ee[now][j] >> shift) & 0xffu;
                const float ws = cf[now][j] * __uint_as_float((eb + 1u) << 23);   // weight x 2^(eb - 126)
                const uint32_t rw[4] = {raw[now][j].x, raw[now][j].y, raw[now][j].z, raw[now][j].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&rw[e]));
                    acc[2 * e] = fmaf(ws, f.x, acc[2 * e]);
                    acc[2 * e + 1] = fmaf(ws, f.y, acc[2 * e + 1]);
                }
            }
        if (row < rows) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 pp = __floats2bfloat162_rn(acc[2 * e], acc[2 * e + 1]);
                w[e] = *reinterpret_cast<const uint32_t *>(&pp);
            }
            *reinterpret_cast<uint4 *>(out + off + sub * 8) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// ------------------------------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    }
    return fn;
}

// The three outer dimensions of K / V (token, head, batch) ordered by ascending stride, as the tensor
// map wants them.  Dimensions of size 1 go last (their stride is never used and is replaced by one that
// keeps the list ascending).  False when two dimensions of size > 1 overlap in memory (a stride of 0 from
// a broadcast view, or a stride smaller than the extent of the dimensions inside it): such a layout is
// not a tiled tensor, and the caller sends it to the generic kernels, which follow any strides.
struct KvDim { unsigned long long size, stride; int which; };
bool order_kv_dims(const Call &c, KvDim (&d)[3]) {
    d[0] = {(unsigned long long)c.Lkv, (unsigned long long)c.kv_st * 2, 0};
    d[1] = {(unsigned long long)c.Hkv, (unsigned long long)c.kv_sh * 2, 1};
    d[2] = {(unsigned long long)c.B, (unsigned long long)c.kv_sb * 2, 2};
    for (int a = 0; a < 3; ++a)
        for (int bq = a + 1; bq < 3; ++bq) {
            const bool swap = (d[bq].size > 1 && d[a].size == 1) ? true
                              : (d[a].size > 1 && d[bq].size == 1) ? false
                              : d[bq].stride < d[a].stride;
            if (swap) { KvDim t = d[a]; d[a] = d[bq]; d[bq] = t; }
        }
    unsigned long long extent = (unsigned long long)kD * 2;   // bytes the dimensions inside cover
    for (int a = 0; a < 3; ++a) {
        if (d[a].size == 1) d[a].stride = extent;
        else if (d[a].stride < extent) return false;
        if (d[a].stride >= (1ull << 40)) return false;        // the tensor map's stride field
        extent = d[a].stride * d[a].size;
    }
    return true;
}

// Tensor map over K or V [B, Hkv, Lkv, 128] with arbitrary nested (16-byte aligned) strides; slot[] says
// where (token, head, batch) ended up among the outer dimensions.
bool make_kv_map(CUtensorMap *tm, const void *ptr, const Call &c, int slot[3]) {
    auto fn = encode_fn();
    if (!fn) return false;
    KvDim d[3];
    if (!order_kv_dims(c, d)) return false;
    for (int a = 0; a < 3; ++a) slot[d[a].which] = a;
    cuuint64_t gdim[4] = {(cuuint64_t)kD, d[0].size, d[1].size, d[2].size};
    cuuint64_t gstr[3] = {d[0].stride, d[1].stride, d[2].stride};
    cuuint32_t box[4] = {64, 1, 1, 1};
    box[1 + slot[0]] = kBK;
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(ptr), gdim, gstr, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Q as rows of 128 elements at one common pitch (the greatest common divisor of its strides), for the row gather.
// False when rows at that pitch would overlap: the caller then works on a dense copy of Q.
long long gcd_ll(long long a, long long b) { while (b) { const long long t = a % b; a = b; b = t; } return a; }
long long q_pitch(const Call &c) {
    long long g = c.q_st;
    if (c.Hq > 1) g = gcd_ll(g, c.q_sh);
    if (c.B > 1) g = gcd_ll(g, c.q_sb);
    return g;
}
bool q_rows_fit(const Call &c) {
    const long long g = q_pitch(c);
    if (g < kD || g >= (1ll << 39)) return false;
    return ((c.B - 1) * c.q_sb + (c.Hq - 1) * c.q_sh + (c.Lq - 1) * c.q_st) / g < (1ll << 31) - 1;
}
bool make_q_map(CUtensorMap *tm, const void *ptr, const Call &c) {
    auto fn = encode_fn();
    if (!fn) return false;
    const long long g = q_pitch(c);
    cuuint64_t gdim[2] = {(cuuint64_t)kD, (cuuint64_t)(((c.B - 1) * c.q_sb + (c.Hq - 1) * c.q_sh + (c.Lq - 1) * c.q_st) / g + 1)};
    cuuint64_t gstr[1] = {(cuuint64_t)g * 2};
    cuuint32_t box[2] = {64, 1}, estr[2] = {1, 1};
    CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), gdim, gstr, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// A stream of up to 128 pieces counts as a tile: out[0] tiles, out[1] pieces, out[2] sum over tiles of (key blocks
// walked), out[3] sum of pieces x blocks
__global__ void __launch_bounds__(256) tile_stats(const int4 *__restrict__ tiles, const int2 *__restrict__ ranges,
                                                  const int *__restrict__ n_tiles, unsigned long long *out) {
    const int n = *n_tiles;
    unsigned long long a = 0, b = 0, c2 = 0, d = 0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const int cnt = tiles[t].w & 0x1ff;
        const int2 r = ranges[t];
        const int n0 = min(cnt, kHalf), n1 = cnt - n0, w0 = (r.x >> 16) - (r.x & 0xffff), w1 = (r.y >> 16) - (r.y & 0xffff);
        a += cnt; b += w0 + w1; c2 += (unsigned long long)n0 * w0 + (unsigned long long)n1 * w1; d += 1 + (n1 > 0);
    }
    atomicAdd(out, d); atomicAdd(out + 1, a); atomicAdd(out + 2, b); atomicAdd(out + 3, c2);
}

}  // namespace

cudaError_t launch_tile_stats(const TcLast &last, long long *out4_device, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out4_device, 0, 4 * sizeof(long long), st);
    if (e != cudaSuccess) return e;
    tile_stats<<<64, 256, 0, st>>>(last.tiles, last.ranges, last.n_tiles, reinterpret_cast<unsigned long long *>(out4_device));
    return cudaGetLastError();
}

bool tc_attention_shape_ok(const Call &c, int dtype) {
    if (dtype != SLA_BF16 || c.D != kD) return false;
    if (c.kv_st < kD || c.top_k > kMaxTopK || !(c.softmax_scale > 0.f)) return false;
    KvDim d[3];
    if (!order_kv_dims(c, d)) return false;   // overlapping K/V dimensions (broadcast views): generic kernels
    const long long ell = base_len(c, c.q_pos0 + c.Lq - 1);
    long long span_tokens = (long long)(c.back + c.fwd) * ell + 1;
    if (c.window > span_tokens) span_tokens = c.window;
    return span_tokens / kBK + 2 <= kMaxWalk;
}

bool tc_attention_supported(const Call &c, int dtype) {
    return tc_attention_shape_ok(c, dtype) && encode_fn() != nullptr;
}

// Scratch layout for a chunk of Lc query positions; returns total bytes.
TcPlan plan_attention_tc(const Call &c, int Lc, size_t gap) {
    TcPlan p;
    p.Lc = Lc;
    p.n_bg = c.B * c.Hkv;
    p.NB = (int)((c.Lkv + kBK - 1) / kBK);
    const long long ell = base_len(c, c.q_pos0 + c.Lq - 1);
    long long span_tokens = (long long)(c.back + c.fwd) * ell + 1;
    if (c.window > span_tokens) span_tokens = c.window;   // the window is a piece too
    if (span_tokens > c.Lkv) span_tokens = c.Lkv;
    p.nb_single = (int)((span_tokens - 1) / kBK + 2);
    // Pieces of a group are ordered by blocks covered, in as many classes as the CTA-local histogram
    // of the counting sort affords (NB * ncls counters in shared memory): up to 8 for the lengths of a
    // single span and, in union mode, up to 32 more for pieces joined from spans that overlap or touch.
    // A tile walks as many key blocks as its longest piece, so a joined piece may only be as long as the
    // classes can still tell apart: when classes of at most kJoinWidth blocks reach up to the longest
    // joined piece there can be (all spans and the window in one), everything that touches is joined;
    // otherwise the classes are shared between single spans and joined pairs, and a piece stops growing
    // at twice a span (measured on the 262144-token configuration: pairs -4 %, triples +1 %).
    // Pieces are joined only where the list is dense: joined pieces come in many lengths, and a stream of 128
    // pieces can only be filled with one of them when the pieces of one end block and class are about that many.
    // `density` is the most pieces an end block (of one batch and KV head) can have on average.  Joined against not
    // joined: density 67 (4096 rows at position 500000, 16 spans of 2049 keys) walks 204 k key blocks against 141 k,
    // for 10 % fewer partials: search and attention 5.02 against 3.97 ms; density 45 (8112 rows at 354345) 3.55
    // against 2.85 ms; density 511 over planted spans 559 against 603 us.  With anchors spread evenly the walk is
    // 5 % shorter without joining at density 417, 2 % at 512 and longer from 2048 on.
    constexpr long long kJoinDensity = 384;
    const long long density = (long long)c.G * Lc * (c.top_k + (c.window > 0 ? 1 : 0)) / p.NB;
    constexpr int kJoinWidth = 3;
    const int ncls_avail = (int)(tc::kHistBytes / ((size_t)p.NB * 4));
    p.ncls1 = p.nb_single < 8 ? p.nb_single : 8;
    while (p.ncls1 > 1 && p.ncls1 > ncls_avail) p.ncls1 /= 2;
    int ncls2 = 0;
    p.nb_max = p.nb_single;
    if (c.mode == SLA_UNION && ncls_avail > p.ncls1 && density >= kJoinDensity) {
        long long joined = (long long)c.top_k * ((long long)(c.back + c.fwd) * ell + 1) + c.window;
        if (joined > c.Lkv) joined = c.Lkv;
        long long nb_full = (joined - 1) / kBK + 2;
        if (nb_full > kMaxWalk) nb_full = kMaxWalk;
        const long long extra = nb_full - p.nb_single;
        const int avail2 = ncls_avail - p.ncls1 < 32 ? ncls_avail - p.ncls1 : 32;
        if (extra > 0 && extra <= (long long)kJoinWidth * avail2) {
            ncls2 = (int)((extra + kJoinWidth - 1) / kJoinWidth);   // fewer classes: fewer global counter updates
            p.nb_max = (int)nb_full;
        } else if (extra > 0 && ncls_avail >= 4) {
            if (p.ncls1 > ncls_avail / 2) p.ncls1 = ncls_avail / 2;
            const int want2 = (p.nb_single + kJoinWidth - 1) / kJoinWidth;
            ncls2 = ncls_avail - p.ncls1 < want2 ? ncls_avail - p.ncls1 : want2;
            if (ncls2 > 32) ncls2 = 32;
            p.nb_max = 2LL * p.nb_single < nb_full ? 2 * p.nb_single : (int)nb_full;
        }
    }
    p.merge_cap = ncls2 > 0 ? (p.nb_max - 2) * kBK : 0;   // a piece of T tokens covers at most (T-1)/64 + 2 blocks
    p.ncls = p.ncls1 + ncls2;
    p.ok = (size_t)p.NB * p.ncls * 4 <= tc::kHistBytes;
    // the work-list kernels hold one CTA per SM (their histogram fills the shared memory): no more CTAs
    // than SMs, or the last few would run as a second wave
    p.ctas_per_bg = 148 / p.n_bg > 1 ? 148 / p.n_bg : 1;
    const size_t rows = (size_t)c.B * c.Hq * Lc;
    p.slots = c.top_k + (c.window > 0 ? 1 : 0);
    const size_t slots = rows * p.slots;
    const size_t n_keys = (size_t)p.n_bg * p.NB * p.ncls;
    // every (batch, kv head) list is cut every kRows records (one ragged tile each) and split again
    // between end blocks (fewer than NB per list)
    p.max_tiles = (long long)(slots / kRows) + (long long)p.n_bg * (p.NB + 1) + 1;
    if (p.max_tiles < kMinTiles) p.max_tiles = kMinTiles;   // every CTA reads its first entry before it knows the count
    size_t off = 0;
    // a region of `size` bytes at the next 256-byte boundary, with a canary gap before it when asked for
    auto take = [&](size_t size) {
        if (gap) { p.canaries.add(off); off += gap; }
        const size_t at = off;
        off = align256(off + size);
        return at;
    };
    p.off_counters = take(64 + (size_t)p.n_bg * 8);
    // the two bucket tables are cleared together at the start of every chunk: no gap between them
    p.off_key_count = take(2 * align256(n_keys * 4));
    p.off_key_cursor = p.off_key_count + align256(n_keys * 4);
    p.off_cta_hist = take((size_t)p.ctas_per_bg * n_keys * 4);
    p.off_tiles = take((size_t)p.max_tiles * 16);
    p.off_ranges = take((size_t)p.max_tiles * 8);
    p.off_recs = take(slots * 16);
    p.off_npieces = take(rows);
    p.off_part_lse = take(slots * 8);
    p.off_part_o = take(slots * kD * 2);
    p.off_q = take(q_rows_fit(c) ? 0 : rows * kD * 2);
    if (gap) { p.canaries.add(off); off += gap; }
    p.bytes = off;
    return p;
}

cudaError_t launch_attn_tc(const void *q, const void *k, const void *v, const Call &c, const int32_t *anchor,
                           const float *score, void *out, float *lse, float *lse_span, void *scratch, size_t scratch_bytes, int sm_count,
                           cudaStream_t st, long long *launches, KernelTimer *timer, bool canaries, TcLast *last) {
    // the largest chunk of query positions whose scratch fits
    const size_t gap = canaries ? Canaries::kBytes : 0;
    long long Lc = c.Lq;
    TcPlan plan = plan_attention_tc(c, (int)Lc, gap);
    while (plan.bytes > scratch_bytes && Lc > 1) {
        Lc = (Lc + 1) / 2;
        plan = plan_attention_tc(c, (int)Lc, gap);
    }
    if (plan.bytes > scratch_bytes || !plan.ok) return cudaErrorMemoryAllocation;
    if (plan.max_tiles > (1ll << 30) || (long long)c.B * c.Hq * Lc * plan.slots > (1ll << 31) - 1) return cudaErrorInvalidValue;

    CUtensorMap tm_q, tm_k, tm_v;
    int slot[3];
    if (!make_kv_map(&tm_k, k, c, slot) || !make_kv_map(&tm_v, v, c, slot)) return cudaErrorInvalidValue;
    const bool q_copied = !q_rows_fit(c);
    if (!q_copied && !make_q_map(&tm_q, q, c)) return cudaErrorInvalidValue;
    // function attributes belong to a device's context: remember them per device, not per process
    static bool attr_set[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(tc_attend<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(tc_attend<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    char *ws = (char *)scratch;
    int *counters = (int *)(ws + plan.off_counters);
    for (long long r0 = 0; r0 < c.Lq; r0 += Lc) {
        const int lc = (int)((c.Lq - r0 < Lc) ? c.Lq - r0 : Lc);
        const long long rows = (long long)c.B * c.Hq * lc;
        cudaError_t e = cudaSuccess;
        if (canaries && (e = launch_canary_fill(ws, plan.canaries, st)) != cudaSuccess) return e;
        tc::PrepArgs pa;
        pa.anchor = anchor; pa.B = c.B; pa.Hq = c.Hq; pa.Hkv = c.Hkv; pa.G = c.G; pa.top_k = c.top_k;
        pa.span_len = c.span_len; pa.back = c.back; pa.fwd = c.fwd; pa.Lq = c.Lq; pa.q_pos0 = c.q_pos0;
        pa.window = c.window; pa.mode = c.mode; pa.len_first = c.len_first; pa.n_len = c.n_len;
        pa.r0 = r0; pa.Lc = lc; pa.NB = plan.NB; pa.nb_max = plan.nb_max; pa.ncls = plan.ncls;
        pa.nb_single = plan.nb_single; pa.ncls1 = plan.ncls1; pa.merge_cap = plan.merge_cap;
        pa.ctas_per_bg = plan.ctas_per_bg;
        pa.key_count = (int *)(ws + plan.off_key_count);
        pa.key_cursor = (int *)(ws + plan.off_key_cursor);
        pa.totals = counters + 16;
        pa.n_tiles = counters;
        pa.ctas = sm_count;
        pa.tiles = (int4 *)(ws + plan.off_tiles);
        pa.ranges = (int2 *)(ws + plan.off_ranges);
        pa.max_tiles = (int)plan.max_tiles;
        pa.recs = (int4 *)(ws + plan.off_recs);
        // the parked pieces borrow the head of the partial-output buffer, which is written only after them
        pa.stage = (int4 *)(ws + plan.off_part_o); pa.slots = plan.slots;
        pa.cta_hist = (int *)(ws + plan.off_cta_hist);
        pa.n_pieces = (unsigned char *)(ws + plan.off_npieces);
        pa.status = c.status;
        e = tc::prepare(pa, st, launches);
        if (e != cudaSuccess) return e;
        TcParams tp;
        if (q_copied) {
            // strides without a common row pitch: the chunk's rows of Q as a dense [B, Hq, lc, 128] tensor
            Call d = c;
            d.Lq = lc; d.q_st = kD; d.q_sh = (long long)lc * kD; d.q_sb = d.q_sh * c.Hq;
            bf16 *qd = (bf16 *)(ws + plan.off_q);
            e = launch_chained(copy_q_rows, dim3((unsigned)((rows * 16 + 255) / 256)), dim3(256), 0, st, (const bf16 *)q, c, r0, lc, qd);
            if (e != cudaSuccess) return e;
            if (launches) *launches += 1;
            if (!make_q_map(&tm_q, qd, d)) return cudaErrorInvalidValue;
            tp.q = qd; tp.q_pitch = kD;
            tp.q_b = c.Hq * lc; tp.q_h = lc; tp.q_t = 1; tp.r0 = 0;
        } else {
            const long long g = q_pitch(c);
            tp.q = (const bf16 *)q; tp.q_pitch = g;
            tp.q_b = (int)(c.B > 1 ? c.q_sb / g : 0); tp.q_h = (int)(c.Hq > 1 ? c.q_sh / g : 0); tp.q_t = (int)(c.q_st / g);
            tp.r0 = (int)r0;
        }
        tp.Hq = c.Hq; tp.Lc = lc; tp.slots = plan.slots;
        tp.scale2 = c.softmax_scale * kLog2e;
        tp.slot_t = slot[0]; tp.slot_h = slot[1]; tp.slot_b = slot[2];
        tp.recs = pa.recs; tp.tiles = pa.tiles; tp.ranges = pa.ranges;
        tp.n_tiles = counters;
        tp.part_o = (__half *)(ws + plan.off_part_o); tp.part_lse = (float2 *)(ws + plan.off_part_lse);
        tp.status = c.status; tp.Hkv = c.Hkv;
        if (last) { last->tiles = pa.tiles; last->ranges = pa.ranges; last->n_tiles = counters; }
        if (timer) timer->begin(st);
        const bool claim = rows * plan.slots >= (long long)kClaimTiles * kRows * sm_count &&
                           plan.nb_single >= (plan.merge_cap > 0 ? kClaimBlocksJoined : kClaimBlocks);
        e = launch_chained(claim ? tc_attend<true> : tc_attend<false>, dim3(sm_count), dim3(kThreads), kSmemBytes, st, tm_q, tm_k, tm_v, tp);
        if (e != cudaSuccess) return e;
        if (timer) timer->end(st);
        // The merges do not release what comes after them: 131072 short CTAs, each with the extra instruction, took 2 % more of
        // a whole call at 65536 positions.  Nor does the search, whose CTAs are in the way of nothing that could start early.
        const unsigned mblocks = (unsigned)((rows * 16 + 255) / 256);
        if (c.mode == SLA_PER_SPAN && c.top_k <= kGateK)
            e = launch_chained(c.top_k <= 2 ? tc_merge_gated_rows<2> : c.top_k <= 4 ? tc_merge_gated_rows<4> : tc_merge_gated_rows<kGateK>, dim3((unsigned)((rows + 255) / 256)), dim3(256), 0, st, (const __half *)tp.part_o,
                               (const float2 *)tp.part_lse, anchor, score, c, plan.slots, lc, r0, (bf16 *)out, lse, lse_span);
        else if (c.mode == SLA_PER_SPAN)
            e = launch_chained(tc_merge_gated, dim3(mblocks), dim3(256), 0, st, (const __half *)tp.part_o, (const float2 *)tp.part_lse,
                               anchor, score, c, plan.slots, lc, r0, (bf16 *)out, lse, lse_span);
        else if (rows < (long long)kMergeFill * sm_count * kMergeLeast || plan.slots * kMergeLeast > kMergePieces)
            e = launch_chained(tc_merge_few, dim3(mblocks), dim3(256), 0, st, (const __half *)tp.part_o, (const float2 *)tp.part_lse,
                               (const unsigned char *)pa.n_pieces, c, plan.slots, lc, r0, (bf16 *)out, lse);
        else {
            int per_warp = 32;
            while (per_warp * plan.slots > kMergePieces || rows < (long long)kMergeFill * sm_count * per_warp) per_warp /= 2;
            const int per_cta = per_warp * kMergeWarps;
            e = launch_chained(tc_merge, dim3((unsigned)((rows + per_cta - 1) / per_cta)), dim3(32 * kMergeWarps),
                               (size_t)per_cta * (plan.slots | 1) * sizeof(float2), st, (const __half *)tp.part_o, (const float2 *)tp.part_lse,
                               (const unsigned char *)pa.n_pieces, c, plan.slots, lc, r0, per_warp, (bf16 *)out, lse);
        }
        if (e != cudaSuccess) return e;
        if (launches) *launches += 2;
        if (canaries && (e = launch_canary_check(ws, plan.canaries, c.status, st)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace sla
