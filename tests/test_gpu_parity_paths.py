"""GPU parity at the sizes where a kernel or a dispatch rule changes over, against the fp64 oracle."""
import pytest

from test_gpu_parity_small import run_prefill, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sla():
    import paper_2601_18401_b200 as sla_pkg
    return sla_pkg


@pytest.fixture(scope="module")
def handle(sla):
    h = sla.Handle(0, 1 << 30)
    sla.sla_set_debug_canaries(h, True)
    yield h
    h.close()


@pytest.mark.parametrize("rows", [1, 130, 382, 383, 384, 900])
def test_pieces_joined_or_not(sla, handle, rows):
    """A chunk at the end of 6144 positions with four query heads per KV head and eight spans: 4 * 8 * rows / 96
    pieces can end in a key block, so that touching spans are joined to one piece from 1152 rows on only; the
    rows of a whole sequence are joined."""
    w = workload(n_q_heads=8, n_kv_heads=2, seq_len=6144, span_len=70, top_k=8, planted_spans=2)
    run_prefill(sla, handle, w, q_pos0=6144 - 3 * rows, Lq=3 * rows)


@pytest.mark.parametrize("seq_len", [127, 128, 129, 255, 256, 257, 384, 385])
def test_streams_of_a_tile(sla, handle, seq_len):
    """One piece per row: tiles whose second stream of 128 pieces is missing, has one piece or is full."""
    run_prefill(sla, handle, workload(n_q_heads=1, n_kv_heads=1, seq_len=seq_len, top_k=1, span_len=40))


@pytest.mark.parametrize("seq_len", [364, 434, 664, 964, 1264])
def test_tiles_dealt_to_a_block(sla, handle, seq_len):
    """Short walks, up to four tiles a block on 148 multiprocessors, each (batch, KV head) ending in a ragged tile: rows of the
    second stream that are copied one and two tiles ahead, or are not there.  (Several spans, from position 64 on: rows of a
    handful of keys may be further off than the tolerance, see test_merge_of_pieces.)"""
    run_prefill(sla, handle, workload(n_q_heads=32, n_kv_heads=8, seq_len=seq_len, top_k=4, span_len=9, seed=79), q_pos0=64)


@pytest.mark.parametrize("span_len", [10, 31, 32, 33, 600])
def test_walks_of_one_block_and_of_many(sla, handle, span_len):
    """Spans within a block, over one boundary and over nineteen blocks; two batches, three KV heads."""
    run_prefill(sla, handle, workload(batch=2, n_q_heads=6, n_kv_heads=3, seq_len=1930, top_k=2, span_len=span_len, seed=78))


def test_query_strides_without_a_common_row_pitch(sla, handle):
    """Heads that start 8 elements after a multiple of the token stride (the rows of Q cannot be numbered at one
    pitch of 128 elements or more), and token rows of 136 elements: same results as on dense tensors."""
    import torch
    from paper_2601_18401_b200 import synth
    w = workload(batch=2, seq_len=700, span_len=30, top_k=3)
    x = synth.make_prefill(w, device="cuda:0")
    B, H, L, D = x["q"].shape
    params = sla.make_params(w.top_k, w.span_len, head_dim=D)
    anchor, _ = sla.sla_span_search(handle, x["q_s"], x["k"], params)
    out, lse = sla.sla_span_attention(handle, x["q"], x["k"], x["v"], anchor, params)
    for st, sh in ((D, L * D + 8), (D + 8, L * (D + 8) + 8)):
        q = torch.zeros(B * H * sh, dtype=x["q"].dtype, device="cuda").as_strided((B, H, L, D), (H * sh, sh, st, 1))
        q.copy_(x["q"])
        out2, lse2 = sla.sla_span_attention(handle, q, x["k"], x["v"], anchor, params)
        torch.cuda.synchronize()
        assert sla.sla_poll_status(handle) == sla.SLA_OK
        assert torch.equal(out2.contiguous(), out) and torch.equal(lse2, lse)


@pytest.mark.parametrize("batch,heads,kv_heads,L", [(1, 4, 1, 1), (1, 8, 2, 17), (2, 6, 3, 1500), (1, 32, 8, 2600)])
def test_query_strides_in_chunks(sla, batch, heads, kv_heads, L):
    """Tokens of all heads side by side with eight elements of padding (no common row pitch): the rows of Q are brought
    together by one kernel per chunk, in a workspace that takes the call at once and in one that takes 1024 rows."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(21)
    D, st = 128, heads * 128 + 8
    q = torch.empty(batch * L * st, dtype=torch.bfloat16, device="cuda").normal_(generator=g).as_strided((batch, heads, L, D), (L * st, D, st, 1))
    k, v = (torch.empty(batch, kv_heads, L, D, dtype=torch.bfloat16, device="cuda").normal_(generator=g) for _ in range(2))
    params = sla.make_params(3, 20, head_dim=D)
    results, launches = [], []
    dense = q.clone(memory_format=torch.contiguous_format)
    for x, rows in ((dense, L), (q, L), (dense, min(L, 1024)), (q, min(L, 1024))):
        h = sla.Handle(0, sla.sla_workspace_bytes(sla.make_layout(x, k), params, rows, L))
        anchor, _ = sla.sla_span_search(h, x, k, params)
        n0 = sla.sla_kernel_launches(h)
        out, lse = sla.sla_span_attention(h, x, k, v, anchor, params)
        launches.append(sla.sla_kernel_launches(h) - n0)
        torch.cuda.synchronize()
        assert sla.sla_poll_status(h) == sla.SLA_OK
        results.append((out.contiguous(), lse))
        h.close()
    for (out, lse), (want, want_lse), n, n_dense in zip(results[1::2], results[::2], launches[1::2], launches[::2]):
        assert torch.equal(out, want) and torch.equal(lse, want_lse)
        assert n_dense % 7 == 0 and n == n_dense // 7 * 8
    assert launches[0] == 7 and (launches[2] > 7) == (L > 1024)


def test_end_blocks_far_apart(sla, handle):
    """Anchors in two narrow regions and in a few places between them: tiles are cut where neighbouring pieces of
    the work list end further apart than a span is long, and streams of one tile walk different key blocks."""
    import parity_util as P
    import torch
    from oracle import sla_oracle as O
    from paper_2601_18401_b200 import synth
    L, top_k, span_len = 9000, 3, 90
    w = workload(n_q_heads=2, n_kv_heads=1, seq_len=L, span_len=span_len, top_k=top_k)
    x = synth.make_prefill(w, device="cuda:0")
    g = torch.Generator().manual_seed(5)
    i = torch.arange(L)[None, None, :, None]
    shape = (1, 2, L, top_k)
    place = torch.randint(0, 10, shape, generator=g)
    spot = torch.where(place < 5, torch.randint(300, 420, shape, generator=g), torch.randint(8000, 8100, shape, generator=g))
    spot = torch.where(place == 9, torch.randint(0, 6, shape, generator=g) * 1000 + 1500, spot)
    anchor = torch.where(spot <= i, spot, torch.full(shape, -1)).to(torch.int32).cuda()
    params = sla.make_params(top_k, span_len, head_dim=128)
    out, lse = sla.sla_span_attention(handle, x["q"], x["k"], x["v"], anchor, params)
    torch.cuda.synchronize()
    assert sla.sla_poll_status(handle) == sla.SLA_OK
    ref = P.oracle_attention_for(P.host_inputs(x), O.BF16, anchor.cpu().numpy(), w)
    P.compare_attention(out, lse, ref, "bf16")


@pytest.mark.parametrize("rows,top_k,span_len", [(1, 1, 0), (40, 2, 0), (40, 1, 300), (257, 2, 0), (33, 3, 5)])
def test_few_rows_far_into_a_context(sla, handle, rows, top_k, span_len):
    """Pieces that lie far apart without a gap longer than a span: a short list is cut into stretches of end blocks, and no
    part walks much more than its stretch and a span."""
    w = workload(n_q_heads=4, n_kv_heads=1, seq_len=60000, top_k=top_k, span_len=span_len)
    run_prefill(sla, handle, w, q_pos0=60000 - rows, Lq=rows)
    span = 2 * (span_len or 245) // 64 + 2
    stats = sla.sla_attention_tile_stats(handle)
    assert 0 < stats["tile_blocks"] <= (max(16, 3 * span) + span) * stats["tiles"]


@pytest.mark.parametrize("heads,kv_heads,top_k", [(8, 1, 1), (16, 2, 4), (16, 1, 8), (16, 1, 16), (8, 1, 13)])
def test_search_of_wide_groups(sla, handle, heads, kv_heads, top_k):
    """Groups of 8 and 16 query heads per KV head, four lanes a head: 1 to 64 strides a row, so that lists of a
    lane stay empty, short or full and the last step of eight or sixteen strides is ragged; lengths not a multiple
    of the positions of a block."""
    import parity_util as P
    import torch
    from oracle import sla_oracle as O
    from paper_2601_18401_b200 import synth
    for batch, seq_len, pos0 in ((1, 1100, 0), (2, 4103, 4062)):
        w = workload(batch=batch, n_q_heads=heads, n_kv_heads=kv_heads, seq_len=seq_len, top_k=top_k, span_len=12)
        x = synth.make_prefill(w, device="cuda:0")
        q_s = x["q_s"][:, :, pos0:]
        anchor, score = sla.sla_span_search(handle, q_s, x["k"], sla.make_params(top_k, 12, head_dim=128), q_pos0=pos0)
        torch.cuda.synchronize()
        host = P.host_inputs({"q_s": q_s, "k": x["k"]})
        ref = O.span_search(host["q_s"], host["k"], synth.dtype_code("bf16"), top_k=top_k, q_pos0=pos0, search_scale=1.0)
        P.compare_search(anchor, score, ref, q_pos0=pos0, q_s=host["q_s"], k=host["k"], search_scale=1.0)


@pytest.mark.parametrize("heads,top_k", [(8, 1), (8, 2), (16, 4), (16, 8), (8, 16), (4, 1), (4, 2), (4, 4), (4, 8), (4, 16)])
def test_search_of_scores_that_are_not_finite(sla, handle, heads, top_k):
    """Keys that hold Inf or NaN, groups of 4, 8 and 16 query heads: a NaN score is no candidate and costs no other one its
    place, -inf comes last, ties go to the nearer anchor."""
    import torch
    L = 430
    g = torch.Generator().manual_seed(13)
    q, k = ((torch.randn(1, h, L, 128, generator=g) * 64).round() / 64 for h in (heads, 1))
    k[0, 0, 50::7] = float("nan")
    k[0, 0, 100, 3], k[0, 0, 200, 9], k[0, 0, 2, 3], k[0, 0, 0, 3] = (float(x) for x in ("-inf", "inf", "inf", "-inf"))
    anchor, score = sla.sla_span_search(handle, q.bfloat16().cuda(), k.bfloat16().cuda(), sla.make_params(top_k, 8, head_dim=128))
    torch.cuda.synchronize()
    anchor, score = anchor.cpu(), score.cpu()
    q, k = q.bfloat16().double(), k.bfloat16().double()
    for i in range(L):
        t = torch.tensor([i + 1 - s * s for s in range(1, i + 2) if s * s <= i + 1])
        x = torch.einsum("hd,td->ht", q[0, :, i], k[0, 0, t])   # multiples of 2^-12 below 2^9: exact in any order
        for h in range(heads):
            keep = ~torch.isnan(x[h])
            order = torch.sort(x[h][keep], descending=True, stable=True).indices[:top_k]
            n = len(order)
            assert torch.equal(anchor[0, h, i, :n].long(), t[keep][order]) and torch.equal(score[0, h, i, :n], x[h][keep][order].float()), (h, i)
            assert (anchor[0, h, i, n:] == -1).all() and torch.isneginf(score[0, h, i, n:]).all()


@pytest.mark.parametrize("heads,kv_heads,seq_len,top_k,window", [
    (32, 8, 2877, 2, 0), (32, 8, 1473, 8, 0), (32, 8, 773, 16, 0),   # 32, 16 and 8 rows a warp, the last warp's cut off
    (32, 8, 417, 6, 40), (16, 4, 417, 4, 0), (1, 1, 101, 3, 0), (2, 1, 579, 64, 100),
])
def test_merge_of_pieces(sla, handle, heads, kv_heads, seq_len, top_k, window):
    """Rows of a warp from 2 to 32, rows that fill no whole block, 2 to 65 slots a row and rows of a single piece.  (From position
    64 on: a row of a handful of keys may be off by 2^-9 (|out| + max |v|), the roundings of the result and of its weights,
    which is more than the tolerance where both are near 4.)"""
    from test_gpu_parity_modes import run_modes
    w = workload(n_q_heads=heads, n_kv_heads=kv_heads, seq_len=seq_len, top_k=top_k, span_len=7)
    if window:
        run_modes(sla, handle, w, window, q_pos0=64)
    else:
        run_prefill(sla, handle, w, q_pos0=64)


@pytest.mark.parametrize("seq_len", [174720, 174721])
def test_buckets_of_the_sort(sla, handle, seq_len):
    """Spans of 81 keys, three length classes: 8190 and 8193 buckets, on both sides of the scan's way of reading them; rows
    that fill no warp of the passes over the pieces."""
    run_prefill(sla, handle, workload(n_q_heads=4, n_kv_heads=2, seq_len=seq_len, top_k=5, span_len=40), q_pos0=seq_len - 301, Lq=301)


@pytest.mark.parametrize("heads,kv_heads,rows,q_pos0,top_k,span_len", [
    (8, 2, 3, 9000, 64, 40), (32, 8, 37, 9000, 64, 40), (8, 1, 1, 9000, 40, 20),   # a few rows a block, some blocks without any
    (32, 8, 37, 9000, 4, 40), (32, 8, 37, 9000, 5, 40),   # pieces that one thread moves in a step, and one more
    (32, 8, 1534, 9000, 5, 40), (32, 8, 1535, 9000, 5, 40),   # 341 and 342 rows a block on 148 multiprocessors
])
def test_rows_of_many_pieces_moved_by_several_threads(sla, handle, heads, kv_heads, rows, q_pos0, top_k, span_len):
    """Rows whose pieces several threads of the list's last pass move, up to 64 pieces a row."""
    run_prefill(sla, handle, workload(n_q_heads=heads, n_kv_heads=kv_heads, seq_len=q_pos0 + rows, top_k=top_k, span_len=span_len), q_pos0=q_pos0)


@pytest.mark.parametrize("heads,top_k", [(4, 2), (4, 16), (8, 16), (16, 16)])
def test_search_beside_a_first_key_that_is_not_finite(sla, handle, heads, top_k):
    """Positions with 131 strides, none of which reaches key 0: an Inf there, with which strides that a position does not have are
    padded, changes nothing and sends no row through the selection pass by pass (four searches 0.1 ms, 0.24 to 1.6 ms where all
    rows took that)."""
    import torch
    L, pos0 = 17423, 131 * 131
    g = torch.Generator(device="cuda").manual_seed(17)
    q, k = (torch.empty(1, h, n, 128, dtype=torch.bfloat16, device="cuda").normal_(generator=g) for h, n in ((heads, L - pos0), (1, L)))
    odd = k.clone()
    odd[:, :, 0, 5] = float("inf")
    params = sla.make_params(top_k, 8, head_dim=128)

    def search(keys):
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                got = sla.sla_span_search(handle, q, keys, params, q_pos0=pos0)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return got, min(times)

    (anchor, score), t = search(k)
    (anchor2, score2), t2 = search(odd)
    assert torch.equal(anchor, anchor2) and torch.equal(score, score2)
    assert t2 < 1.5 * t, (t, t2)


def test_lists_around_the_plain_shared_memory():
    """Eight length classes and 1531 to 1536 key blocks: histograms of 48992 to 49168 bytes (with the class table), around the 48 KB
    that a kernel has without asking, of which its own arrays are a part.  In a process of its own, the smallest first: what a
    longer list was allowed before would hide a size that is not asked for."""
    import os
    import subprocess
    import sys
    code = """if True:
        import paper_2601_18401_b200 as sla
        from test_gpu_parity_modes import run_modes
        from test_gpu_parity_small import run_prefill, workload
        h = sla.Handle(0, 256 << 20)
        sla.sla_set_debug_canaries(h, True)
        for L in (97984, 97985, 98240, 98241):
            w = workload(n_q_heads=4, n_kv_heads=1, seq_len=L, top_k=8, span_len=0)
            run_prefill(sla, h, w, q_pos0=L - 301)
            run_modes(sla, h, w.scaled(top_k=2, back_factor=4, fwd_factor=2), 1088, q_pos0=L - 301)
        """
    here = os.path.dirname(os.path.abspath(__file__))
    path = os.pathsep.join([here, os.path.dirname(here), os.environ.get("PYTHONPATH", "")])
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, PYTHONPATH=path), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("window", [0, 1, 24, 25, 400, 2**31 - 1])
@pytest.mark.parametrize("heads", [4, 8, 16])
def test_search_walk_of_strides(sla, handle, heads, window):
    """Groups of 4, 8 and 16 query heads at lengths around the positions of a warp and of a block, windows that leave all,
    some or no strides (the largest has a stride whose square exceeds 31 bits); scores exact in any order of summation."""
    import torch
    g = torch.Generator().manual_seed(29)
    for L, pos0, top_k in ((1, 0, 1), (3, 0, 2), (5, 0, 8), (15, 2, 4), (17, 0, 16), (33, 30, 8), (402, 380, 4), (1100, 1059, 16)):
        q, k = ((torch.randn(1, h, n, 128, generator=g) * 64).round() / 64 for h, n in ((heads, L - pos0), (1, L)))
        q, k = q.bfloat16(), k.bfloat16()
        params = sla.make_params(top_k, 8, window=window, head_dim=128)
        anchor, score = sla.sla_span_search(handle, q.cuda(), k.cuda(), params, q_pos0=pos0)
        torch.cuda.synchronize()
        anchor, score, q, k = anchor.cpu(), score.cpu(), q.double(), k.double()
        for i in range(pos0, L):
            t = torch.tensor([i + 1 - s * s for s in range(1, i + 2) if window < s * s <= i + 1], dtype=torch.long)
            x = torch.einsum("hd,td->ht", q[0, :, i - pos0], k[0, 0, t])
            order = torch.sort(x, dim=1, descending=True, stable=True).indices[:, :top_k]
            n = order.shape[1]
            a, v = anchor[0, :, i - pos0], score[0, :, i - pos0]
            assert torch.equal(a[:, :n].long(), t[order]) and torch.equal(v[:, :n], x.gather(1, order).float()), (L, i)
            assert (a[:, n:] == -1).all() and torch.isneginf(v[:, n:]).all()


@pytest.mark.parametrize("dtype,top_k", [("f32", 1), ("f32", 9), ("bf16", 64)])
def test_generic_search_of_equal_scores(sla, handle, dtype, top_k):
    """Small whole numbers, zeros of both signs among the products: many equal scores, the nearer anchor first, for fewer and
    more strides than lanes."""
    import torch
    L, g = 1700, torch.Generator().manual_seed(31)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    q, k = (torch.zeros(1, 1, L, 64) for _ in range(2))
    q[..., :3], k[..., :3] = (torch.randint(-1, 2, (1, 1, L, 3), generator=g).float() for _ in range(2))
    k[:, :, ::5] = -0.0
    anchor, score = sla.sla_span_search(handle, q.to(dt).cuda(), k.to(dt).cuda(), sla.make_params(top_k, 8, head_dim=64))
    torch.cuda.synchronize()
    anchor, score = anchor.cpu()[0, 0], score.cpu()[0, 0]
    for i in range(0, L, 7):
        t = torch.tensor([i + 1 - s * s for s in range(1, i + 2) if s * s <= i + 1])
        x = k[0, 0, t] @ q[0, 0, i]
        order = torch.sort(x, descending=True, stable=True).indices[:top_k]
        n = len(order)
        assert torch.equal(anchor[i, :n].long(), t[order]) and torch.equal(score[i, :n], x[order]), i
        assert (anchor[i, n:] == -1).all() and torch.isneginf(score[i, n:]).all()


@pytest.mark.parametrize("heads,kv_heads,seq_len,top_k", [
    (32, 8, 415, 4), (32, 8, 416, 4), (32, 8, 416, 32), (32, 8, 416, 33), (32, 8, 416, 64), (2, 1, 164, 64)])
def test_merge_of_few_rows(sla, handle, heads, kv_heads, seq_len, top_k):
    """Rows and slots on both sides of the numbers up to which a warp merges several rows (11248 rows on 148 multiprocessors, 32 slots), four rows a
    warp.  (From position 64 on, see test_merge_of_pieces.)"""
    run_prefill(sla, handle, workload(n_q_heads=heads, n_kv_heads=kv_heads, seq_len=seq_len, top_k=top_k, span_len=7), q_pos0=64)


@pytest.mark.parametrize("by_blocks,kw", [
    # few keys a row, few rows (at the start, or far into a context), or blocks that few rows select
    (False, dict(seq_len=1, top_k=6, span_len=300)), (False, dict(seq_len=65, top_k=64, span_len=2)),
    (False, dict(seq_len=900, top_k=1, span_len=31)), (False, dict(seq_len=60020, q_pos0=60000, span_len=16)),
    (False, dict(seq_len=9000, q_pos0=8744, top_k=16, span_len=4)),
    # a last block of 63, 64 keys and one key
    (True, dict(seq_len=1599, top_k=8, span_len=40)), (True, dict(seq_len=1600, top_k=8, span_len=40)),
    (True, dict(seq_len=1601, top_k=8, span_len=40)),
    (True, dict(batch=2, n_q_heads=6, n_kv_heads=2, seq_len=1543, top_k=9, span_len=0)),   # lists that fill up several times
    # lists of less than a row per group and warp up to more than four: one to four rows per group, one pass and two
    (True, dict(n_q_heads=1, seq_len=4099, top_k=4, span_len=64)), (True, dict(seq_len=2600, top_k=4, span_len=40)),
    (True, dict(seq_len=2300, top_k=6, span_len=33, window=200)), (True, dict(seq_len=3000, q_pos0=2100, top_k=8, span_len=60, window=129)),
    (True, dict(n_q_heads=4, n_kv_heads=4, seq_len=1200, top_k=8, span_len=100)),
    (True, dict(seq_len=1000, span_len=600)), (True, dict(seq_len=700, top_k=64, span_len=40)),   # spans cut off at 0; 64 of them
    (True, dict(seq_len=20000, q_pos0=19301, span_len=0)),
])
@pytest.mark.parametrize("dtype,D", [("f32", 64), ("f32", 128), ("bf16", 64)])
def test_key_blocks(sla, handle, by_blocks, kw, dtype, D):
    """The generic span-attention on both sides of the rule that chooses between the kernels by rows and by blocks of keys,
    against the oracle; and the two kernels against each other (a workspace without room leaves the one by rows), rows
    without any anchor among them."""
    import torch
    from test_gpu_parity_modes import run_modes
    from paper_2601_18401_b200 import synth
    window, q_pos0 = kw.get("window", 0), kw.get("q_pos0", 0)
    w = workload(**dict(dict(n_q_heads=2, n_kv_heads=1), **{n: x for n, x in kw.items() if n not in ("window", "q_pos0")}, dtype=dtype, head_dim=D))
    if window:
        run_modes(sla, handle, w, window, q_pos0=q_pos0)
    else:
        run_prefill(sla, handle, w, q_pos0=q_pos0)
    x = synth.make_prefill(w, device="cuda:0")
    q_s, q = x["q_s"][:, :, q_pos0:], x["q"][:, :, q_pos0:]
    params = sla.make_params(w.top_k, w.span_len, head_dim=D, window=window)
    anchor, _ = sla.sla_span_search(handle, q_s, x["k"], params, q_pos0=q_pos0)
    anchor[:, :, 1::5] = -1
    small = sla.Handle(0, 1024)
    n0, m0 = sla.sla_kernel_launches(handle), sla.sla_kernel_launches(small)
    out, lse = sla.sla_span_attention(handle, q, x["k"], x["v"], anchor, params, q_pos0=q_pos0)
    out2, lse2 = sla.sla_span_attention(small, q, x["k"], x["v"], anchor, params, q_pos0=q_pos0)
    torch.cuda.synchronize()
    # blocks of keys and their merge for every chunk of rows, or the kernel by rows
    assert (sla.sla_kernel_launches(handle) - n0 > 1) == by_blocks and sla.sla_kernel_launches(small) - m0 == 1
    assert sla.sla_poll_status(handle) == sla.SLA_OK and sla.sla_poll_status(small) == sla.SLA_OK
    small.close()
    # both sum the same products and exponentials in fp32 in other orders: at most (D + n_keys + 30) 2^-24 of a score or a sum
    # of |scores| < 64, and for bf16 results a rounding of 2^-8 of values < 5 on either side
    n_keys = min(w.seq_len, w.top_k * (2 * (w.span_len or 142) + 1) + window)
    tol = 64 * (D + n_keys + 30) * 2.0 ** -24 * 0.25 + (5 * 2.0 ** -8 if dtype == "bf16" else 0.0)
    fin = torch.isfinite(lse2)
    assert bool((torch.isfinite(lse) == fin).all())
    assert float((out.double() - out2.double()).abs().max()) <= tol and bool(((lse - lse2)[fin].abs() <= tol).all())


@pytest.mark.parametrize("rows,pos0,kv_heads,D,top_k,span_len,dtype,most", [
    (16, 300000, 8, 128, 4, 32, "f32", 1), (1, 300000, 8, 64, 4, 32, "f32", 1), (256, 60000, 4, 64, 2, 64, "bf16", 1),
    (500, 100000, 2, 128, 4, 447, "f32", 2), (100, 100000, 2, 128, 4, 447, "f32", 2),
])
def test_generic_rows_far_into_a_context(sla, rows, pos0, kv_heads, D, top_k, span_len, dtype, most):
    """A few rows with short spans do not go through all blocks of a long context (they took up to 25 times as long);
    long spans do."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(9)
    T = torch.float32 if dtype == "f32" else torch.bfloat16
    q, k, v = (torch.empty(1, kv_heads, n, D, dtype=T, device="cuda").normal_(generator=g) for n in (rows, pos0 + rows, pos0 + rows))
    params = sla.make_params(top_k, span_len, head_dim=D)
    h = sla.Handle(0, sla.sla_workspace_bytes(sla.make_layout(q, k), params, rows, pos0 + rows))
    anchor, _ = sla.sla_span_search(h, q, k, params, q_pos0=pos0)
    n0 = sla.sla_kernel_launches(h)
    out, _ = sla.sla_span_attention(h, q, k, v, anchor, params, q_pos0=pos0)
    assert sla.sla_kernel_launches(h) - n0 == most and sla.sla_poll_status(h) == sla.SLA_OK and bool(torch.isfinite(out).all())
    h.close()


@pytest.mark.parametrize("dtype,D", [("f32", 64), ("f32", 128), ("bf16", 64)])
def test_values_of_other_rows_do_not_leak(sla, dtype, D):
    """Inf and NaN among the values reach the rows that selected their key and no others: not those that selected
    another key of the block, nor those before it.  The kernels by key blocks and by rows agree on every entry."""
    import math
    import torch
    L, top_k, ell = 1100, 8, 33
    g = torch.Generator().manual_seed(11)
    q, k, v = (torch.randn(1, 2, L, D, generator=g).to(torch.float32 if dtype == "f32" else torch.bfloat16).cuda() for _ in range(3))
    for at, x in {(0, 333, 5): math.nan, (0, 1099, 0): math.inf, (1, 64, D - 1): -math.inf, (1, 64, 2): math.nan, (1, 127, 7): math.inf,
                  (1, 500, 7): -math.inf}.items():
        v[(0, *at)] = x
    params = sla.make_params(top_k, ell, head_dim=D)
    h, small = sla.Handle(0, sla.sla_workspace_bytes(sla.make_layout(q, k), params, L, L)), sla.Handle(0, 1024)
    anchor, _ = sla.sla_span_search(h, q, k, params)
    n0 = sla.sla_kernel_launches(h)
    out, lse = sla.sla_span_attention(h, q, k, v, anchor, params)
    assert sla.sla_kernel_launches(h) - n0 == 2   # blocks of keys, merge
    out2, lse2 = sla.sla_span_attention(small, q, k, v, anchor, params)
    torch.cuda.synchronize()
    assert sla.sla_poll_status(h) == sla.SLA_OK and sla.sla_poll_status(small) == sla.SLA_OK
    h.close()
    small.close()
    # entries of the output that a selected key's value makes non-finite
    i, a = torch.arange(L)[None, None, :, None], anchor.cpu().long()
    j = torch.arange(L)
    sel = torch.zeros(1, 2, L, L, dtype=torch.bool)
    for x in range(top_k):
        t = a[..., x:x + 1]
        sel |= (t >= 0) & (j >= t - 2 * ell) & (j <= torch.minimum(t, i))
    hit = (sel.float() @ (~torch.isfinite(v.cpu())).float()) > 0
    assert torch.equal(~torch.isfinite(out.cpu()), hit) and hit.any() and not hit.all()
    assert torch.equal(torch.isnan(out), torch.isnan(out2)) and torch.equal(torch.isposinf(out), torch.isposinf(out2))
    fin = torch.isfinite(out)
    # as in test_key_blocks: at most (D + L + 30) 2^-24 of sums of |scores| < 64, a bf16 rounding of values < 5
    tol = 64 * (D + L + 30) * 2.0 ** -24 * 0.25 + (5 * 2.0 ** -8 if dtype == "bf16" else 0.0)
    assert (out.double() - out2.double())[fin].abs().max().item() <= tol and (lse - lse2).abs().max().item() <= tol


def test_token_stride_above_31_bits(sla):
    """Tokens 2^31 + 64 elements apart: search and attention read the same rows as on a dense tensor."""
    import torch
    D, L, st = 64, 9, (1 << 31) + 64
    g = torch.Generator().manual_seed(3)
    q, k = (torch.randn(1, 2, L, D, generator=g).bfloat16().cuda() for _ in range(2))
    far = torch.empty((L - 1) * st + 2 * D, dtype=torch.bfloat16, device="cuda").as_strided((1, 2, L, D), (L * st, D, st, 1))
    far.copy_(k)
    params = sla.make_params(2, 2, head_dim=D)
    h = sla.Handle(0, 1 << 20)
    want, got = (sla.sla_span_search(h, q, x, params) for x in (k, far))
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    want, got = (sla.sla_span_attention(h, q, x, x, want[0], params) for x in (k, far))
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert sla.sla_poll_status(h) == sla.SLA_OK
    h.close()


@pytest.mark.parametrize("seq_len,heads,kv_heads", [(1023, 32, 8), (1024, 32, 8), (1025, 32, 8), (4097, 8, 2), (8193, 16, 4)])
def test_host_chunks(sla, seq_len, heads, kv_heads):
    """Prefill through host buffers in chunks that shrink towards the end: one chunk and the first lengths with two, the
    smallest chunk longer than 512 positions with few heads, quarters of the sequence first."""
    import parity_util as P
    import torch
    from paper_2601_18401_b200 import synth
    w = workload(seq_len=seq_len, n_q_heads=heads, n_kv_heads=kv_heads, span_len=24, top_k=5)
    x = synth.make_prefill(w, device="cuda:0")
    params = sla.make_params(w.top_k, w.span_len, head_dim=128)
    layout = sla.make_layout(x["q"], x["k"])
    h = sla.Handle(0, sla.sla_workspace_bytes(layout, params, seq_len, seq_len) + sla.sla_host_staging_bytes(layout, params, seq_len))
    anchor, score = sla.sla_span_search(h, x["q_s"], x["k"], params)
    out, lse = sla.sla_span_attention(h, x["q"], x["k"], x["v"], anchor, params)
    host = {n: t.cpu().pin_memory() for n, t in x.items()}
    ho, hl, ha, hs = sla.sla_prefill_host(h, host["q_s"], host["q"], host["k"], host["v"], params)
    assert sla.sla_poll_status(h) == sla.SLA_OK
    h.close()
    assert torch.equal(ha, anchor.cpu()) and torch.equal(hs, score.cpu())
    # either side is within the tolerance of the exact result (touching spans may be joined on one side only)
    assert (ho.float() - out.cpu().float()).abs().max().item() <= 2 * P.OUT_TOL["bf16"]
    fin = torch.isfinite(lse.cpu())
    assert torch.equal(torch.isfinite(hl), fin) and (hl[fin] - lse.cpu()[fin]).abs().max().item() <= 2 * P.LSE_TOL["bf16"]


@pytest.mark.parametrize("heads", [1, 2, 4])
@pytest.mark.parametrize("spare", [4, 1 << 20, (1 << 20) + 12])
def test_host_staging_in_a_larger_workspace(sla, heads, spare):
    """A handle with more room than asked for and an odd number of rows: the staging buffers start on an aligned address
    all the same, and the kernels are those of the exact size (groups of four: the fused selection, launched once)."""
    import torch
    from paper_2601_18401_b200 import synth
    L = 301
    w = workload(seq_len=L, n_q_heads=heads, n_kv_heads=1, span_len=8, top_k=3)
    x = synth.make_prefill(w, device="cuda:0")
    host = {n: t.cpu().pin_memory() for n, t in x.items()}
    params = sla.make_params(w.top_k, w.span_len, head_dim=128)
    layout = sla.make_layout(x["q"], x["k"])
    need = sla.sla_workspace_bytes(layout, params, L, L) + sla.sla_host_staging_bytes(layout, params, L)
    results, launches = [], []
    for room in (need, need + spare):
        h = sla.Handle(0, room)
        results.append([t.clone() for t in sla.sla_prefill_host(h, host["q_s"], host["q"], host["k"], host["v"], params)])
        assert sla.sla_poll_status(h) == sla.SLA_OK
        launches.append(sla.sla_kernel_launches(h))
        h.close()
    assert launches[0] == launches[1] and all(torch.equal(a, b) for a, b in zip(*results))


@pytest.mark.parametrize("top_k", [1, 2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("window", [0, 40])
def test_gated_merge_of_each_width(sla, handle, top_k, window):
    """The per-span merge is built for up to 2, 4 and 8 spans a row, the counting pass of the work list for up to 5, 9 and
    17 spans and window together; beyond that the general ones."""
    from test_gpu_parity_modes import run_modes
    run_modes(sla, handle, workload(n_q_heads=2, n_kv_heads=1, seq_len=1100, top_k=top_k, span_len=21), window)


@pytest.mark.parametrize("B,Hq,Hkv,dtype,D,n_ctx,top_k,span_len,per_span", [
    (1, 8, 2, "bf16", 128, 70001, 16, 600, False),    # clusters of eight, several per head
    (1, 32, 8, "bf16", 128, 9001, 8, 0, False),       # one cluster of eight per head
    (2, 32, 8, "bf16", 128, 4099, 3, 300, False),     # clusters of four
    (4, 32, 4, "bf16", 64, 4099, 2, 500, False),      # clusters of two, head_dim 64
    (2, 32, 8, "f32", 128, 3001, 2, 700, True),       # per-span units in clusters of two
    (10, 32, 8, "bf16", 128, 16384, 4, 30, False),    # one CTA per head; 128 anchors: it scores them itself
    (10, 32, 8, "bf16", 128, 16641, 4, 30, False),    # 129 anchors: scored first
    (1, 2, 1, "f32", 64, 1050000, 33, 90, False),     # 1024 anchors and one more per CTA of a cluster of eight
    (1, 4, 1, "bf16", 128, 40, 64, 3, False),         # fewer anchors than slots, one CTA per head
])
def test_decode_split_over_clusters(sla, handle, B, Hq, Hkv, dtype, D, n_ctx, top_k, span_len, per_span):
    """Decode steps on both sides of the rule that deals a step to CTAs and clusters; the anchors in a local window
    of 64 tokens are left out in the per-span case."""
    import parity_util as P
    import torch
    from oracle import sla_oracle as O
    from paper_2601_18401_b200 import synth
    w = synth.Workload("dc", "decode", B, Hq, Hkv, D, n_ctx, dtype, span_len, top_k, seed=67)
    kc, vc = synth.make_decode_cache(w, "cuda:0", capacity=n_ctx)
    x = synth.make_decode_step_inputs(w, 0, "cuda:0")
    window = 64 if per_span else 0
    params = sla.make_params(top_k, span_len, window=window, mode=sla.SLA_PER_SPAN if per_span else sla.SLA_UNION, head_dim=D)
    for rep in range(2):   # the second step finds the completion counters as the first left them
        got = sla.sla_decode_step(handle, x["q_s"], x["q"], kc, vc, n_ctx, params)
        torch.cuda.synchronize()
        assert sla.sla_poll_status(handle) == sla.SLA_OK
    P.check_decode_step(got, synth.to_numpy(x["q_s"]), synth.to_numpy(x["q"]), synth.to_numpy(kc), synth.to_numpy(vc),
                        synth.dtype_code(dtype), dtype, n_ctx=n_ctx, top_k=top_k, span_len=span_len, window=window,
                        mode=O.PER_SPAN if per_span else O.UNION)


@pytest.mark.parametrize("n_ctx,Hq,top_k", [(200, 4, 8), (90000, 4, 16), (90000, 4, 64), (66000, 320, 5), (200000, 320, 40)])
def test_decode_equal_scores(sla, handle, n_ctx, Hq, top_k):
    """All scores equal: the nearest anchors win, in order; more candidates than the selection's list holds."""
    import math
    import torch
    k = torch.ones(1, 1, n_ctx, 64, dtype=torch.bfloat16, device="cuda").expand(1, Hq // 4, n_ctx, 64)
    q = torch.ones(1, Hq, 64, dtype=torch.bfloat16, device="cuda")
    _, _, anchor, score = sla.sla_decode_step(handle, q, q, k, k, n_ctx, sla.make_params(top_k, 5, head_dim=64))
    torch.cuda.synchronize()
    assert sla.sla_poll_status(handle) == sla.SLA_OK
    n = min(top_k, math.isqrt(n_ctx))
    want = torch.tensor([n_ctx - (s + 1) ** 2 if s < n else -1 for s in range(top_k)], dtype=torch.int32)
    assert torch.equal(anchor.cpu(), want.expand(1, Hq, top_k))
    assert (score[..., :n] == 64.0).all()
