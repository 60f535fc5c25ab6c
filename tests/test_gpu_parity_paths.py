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
