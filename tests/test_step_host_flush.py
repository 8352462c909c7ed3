"""Host-buffer steps that are flushed one by one (dx leaves under the weight gradients from the second call on) and in
a row: every call returns what the device-resident path computes, in either mode and across the change, with all the
calls in flight at once."""
import pytest
import torch

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth

pytestmark = pytest.mark.gpu

KEPT = ("dW_gate", "dW_down", "dE_rows", "unique_ids", "n_unique")


@pytest.mark.parametrize("wait", [False, True], ids=["in flight", "one at a time"])
@pytest.mark.parametrize("T,d,F", [(300, 136, 264), (5000, 256, 1032)])
def test_flushed_and_unflushed_calls(T, d, F, wait):
    V = 400
    shape = B.make_shape(T, d, F, V, B.DTYPE_BF16, B.DTYPE_FP32, 0)
    arena = torch.empty(B.stem_step_arena_bytes(shape), dtype=torch.uint8, device="cuda")
    B.stem_init_workspace(arena)
    w = synth.Workload("t", T, d, F, V, "bf16", "zipf")
    st = runner.state_from_numpy(synth.make_inputs(w, seed=61), B.DTYPE_BF16, V)
    gen = torch.Generator(device="cuda")
    flushes = (True, True, True, False, False, False, True, True, True, False)
    calls = []
    for i in range(len(flushes)):
        gen.manual_seed(i)
        st.x.normal_(generator=gen)
        st.dy.normal_(generator=gen)
        st.ids.random_(0, V - 37 * i, generator=gen)           # every call has its own count of rows
        st.step()
        torch.cuda.synchronize()
        calls.append({
            "host": {k: getattr(st, k).cpu().pin_memory() for k in ("x", "dy", "ids")},
            "out": {"y": torch.zeros(T, d, dtype=torch.bfloat16).pin_memory(), "dx": torch.zeros(T, d, dtype=torch.bfloat16).pin_memory(),
                    "n": torch.zeros(1, dtype=torch.int32).pin_memory()},
            "dev": {k: torch.zeros_like(st.bufs[k]) for k in KEPT},
            "ref": {k: st.bufs[k].clone() for k in KEPT + ("y", "dx")},
        })
    torch.cuda.synchronize()
    for c, flush in zip(calls, flushes):
        h, o, g = c["host"], c["out"], c["dev"]
        B.stem_ffn_step_host(shape, h["x"], h["ids"], h["dy"], st.W_gate, st.E, st.W_down, o["y"], o["dx"], g["dW_gate"],
                             g["dW_down"], g["dE_rows"], g["unique_ids"], g["n_unique"], o["n"], arena)
        if flush:
            B.stem_ffn_step_host_flush()
        if wait:
            torch.cuda.synchronize()
    B.stem_ffn_step_host_flush()
    torch.cuda.synchronize()
    assert B.stem_query_status(arena) == B.OK
    for i, c in enumerate(calls):
        o, g, ref = c["out"], c["dev"], c["ref"]
        n_u = int(ref["n_unique"].item())
        assert int(o["n"][0]) == n_u == int(g["n_unique"].item()), i
        assert torch.equal(o["y"], ref["y"].cpu()) and torch.equal(o["dx"], ref["dx"].cpu()), i
        for k in ("dW_gate", "dW_down"):
            assert torch.equal(g[k], ref[k]), (i, k)
        for k in ("dE_rows", "unique_ids"):
            assert torch.equal(g[k][:n_u], ref[k][:n_u]), (i, k)
