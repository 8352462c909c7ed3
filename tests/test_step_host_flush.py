"""Host-buffer steps that are flushed one by one (dx leaves under the weight gradients from the second call on) and in
a row: every call returns what the device-resident path computes, in either mode and across the change."""
import pytest
import torch

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,F", [(300, 136, 264), (5000, 256, 1032)])
def test_flushed_and_unflushed_calls(T, d, F):
    V = 400
    shape = B.make_shape(T, d, F, V, B.DTYPE_BF16, B.DTYPE_FP32, 0)
    arena = torch.empty(B.stem_step_arena_bytes(shape), dtype=torch.uint8, device="cuda")
    B.stem_init_workspace(arena)
    w = synth.Workload("t", T, d, F, V, "bf16", "zipf")
    st = runner.state_from_numpy(synth.make_inputs(w, seed=61), B.DTYPE_BF16, V)
    gen = torch.Generator(device="cuda")
    dev = {k: torch.zeros_like(st.bufs[k]) for k in ("dW_gate", "dW_down", "dE_rows", "unique_ids", "n_unique")}
    for i, flush in enumerate((True, True, True, False, False, True, True)):
        gen.manual_seed(i)
        st.x.normal_(generator=gen)
        st.dy.normal_(generator=gen)
        host = {k: getattr(st, k).cpu().pin_memory() for k in ("x", "dy", "ids")}
        out = {"y": torch.zeros_like(host["x"]).pin_memory(), "dx": torch.zeros_like(host["x"]).pin_memory(),
               "n": torch.zeros(1, dtype=torch.int32).pin_memory()}
        B.stem_ffn_step_host(shape, host["x"], host["ids"], host["dy"], st.W_gate, st.E, st.W_down, out["y"], out["dx"],
                             dev["dW_gate"], dev["dW_down"], dev["dE_rows"], dev["unique_ids"], dev["n_unique"], out["n"], arena)
        if flush:
            B.stem_ffn_step_host_flush()
        torch.cuda.synchronize()
        st.step()
        torch.cuda.synchronize()
        n_u = int(st.bufs["n_unique"].item())
        assert B.stem_query_status(arena) == B.OK and int(out["n"][0]) == n_u
        assert torch.equal(out["y"], st.bufs["y"].cpu()) and torch.equal(out["dx"], st.bufs["dx"].cpu()), i
        for k in ("dW_gate", "dW_down"):
            assert torch.equal(dev[k], st.bufs[k]), (i, k)
        assert torch.equal(dev["dE_rows"][:n_u], st.bufs["dE_rows"][:n_u]), i
