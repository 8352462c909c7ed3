"""Which call of stem_ffn_step_host makes dx ahead of the other gradients: the order is the calling thread's own
habit of flushing, whatever other threads do and however often it flushes."""
import threading

import pytest
import torch

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth

pytestmark = pytest.mark.gpu


@pytest.fixture
def call():
    T, d, F, V = 300, 136, 264, 100
    shape = B.make_shape(T, d, F, V, B.DTYPE_BF16, B.DTYPE_FP32, 0)
    st = runner.state_from_numpy(synth.make_inputs(synth.Workload("t", T, d, F, V, "bf16", "zipf"), seed=62), B.DTYPE_BF16, V)
    arena = torch.empty(B.stem_step_arena_bytes(shape), dtype=torch.uint8, device="cuda")
    B.stem_init_workspace(arena)
    host = {k: getattr(st, k).cpu().pin_memory() for k in ("x", "dy", "ids")}
    y, dx = (torch.zeros_like(host["x"]).pin_memory() for _ in range(2))
    b = st.bufs
    torch.cuda.synchronize()

    def one():
        """One call; whether dx came before the table gradient."""
        B.stem_profile_enable(True)
        B.stem_ffn_step_host(shape, host["x"], host["ids"], host["dy"], st.W_gate, st.E, st.W_down, y, dx, b["dW_gate"],
                             b["dW_down"], b["dE_rows"], b["unique_ids"], b["n_unique"], None, arena)
        torch.cuda.synchronize()
        names = [n for n, _ in B.stem_profile_records()]
        B.stem_profile_enable(False)
        return names.index("dx_gemm") < names.index("seg_reduce")

    flush = B.stem_ffn_step_host_flush
    # whatever ran before: two unflushed calls, then a flush, is no habit of flushing every call
    one(), one(), flush()
    yield one, flush
    flush()
    torch.cuda.synchronize()


def test_order_follows_the_flushes(call):
    one, flush = call
    assert not one()
    flush()
    assert one()                    # the last flush followed one call
    assert not one()                # the second call without a flush
    flush()
    assert not one()
    flush()
    assert one()


def test_a_second_flush_in_a_row_changes_nothing(call):
    one, flush = call
    one(), flush(), flush()
    assert one()
    flush(), flush(), flush()
    assert one()


def test_another_threads_calls_change_nothing(call):
    one, flush = call
    one(), flush()
    seen = []
    t = threading.Thread(target=lambda: seen.extend([one(), one()]))
    t.start()
    t.join()
    assert seen == [False, False]   # that thread has not flushed yet
    assert one()
    flush()
    assert one()
