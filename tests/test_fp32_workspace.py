"""fp32 layers in a workspace without room for the three bf16 parts of the operands: what fitted a layer on the FMA
kernels still does, with their results."""
import pytest
import torch

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth


def _bytes(T, d, F, V, flags):
    s = B.make_shape(T, d, F, V, B.DTYPE_FP32, B.DTYPE_FP32, flags)
    return B.stem_workspace_bytes(s), B.stem_step_arena_bytes(s)


@pytest.mark.parametrize("T,d,F,V", [(2048, 1024, 2816, 32000), (256, 256, 688, 4096), (16384, 2048, 8192, 32000)])
def test_the_fma_kernels_need_no_room_for_parts(T, d, F, V):
    tensor = T * F * 4
    ws, arena = _bytes(T, d, F, V, B.FLAG_SIMT)
    # dU and dG, and the partial rows of the table-gradient reduce
    assert 2 * tensor <= ws < 3 * tensor
    more = _bytes(T, d, F, V, 0)
    # three bf16 numbers per element of x, dy, both weights, H and dG, and a word per 4096 of them
    parts = 6 * (2 * T * d + 2 * F * d + 2 * T * F)
    for a, b in zip((ws, arena), more):
        assert a + parts <= b <= a + parts * 1.001 + 16384


def test_a_smaller_one_is_refused():
    import ctypes
    s = B.make_shape(64, 64, 128, 100, B.DTYPE_FP32, B.DTYPE_FP32, 0)
    need, arena = _bytes(64, 64, 128, 100, B.FLAG_SIMT)
    p = 0x10000
    assert B.lib().stem_ffn_forward(ctypes.byref(s), p, p, p, p, p, p, None, None, p, need - 1, None) == B.ERR_WORKSPACE_TOO_SMALL
    args = [ctypes.byref(s)] + [p] * 15 + [p, arena - 1, None]
    assert B.lib().stem_ffn_step_host(*args) == B.ERR_WORKSPACE_TOO_SMALL


@pytest.mark.gpu
@pytest.mark.parametrize("room", ["least", "one byte short of the parts"])
def test_layer_in_a_small_workspace(room):
    T, d, F, V = 333, 132, 268, 120
    least, arena_least = _bytes(T, d, F, V, B.FLAG_SIMT)
    whole, arena_whole = _bytes(T, d, F, V, 0)
    n, n_arena = (least, arena_least) if room == "least" else (whole - 1, arena_whole - 1)
    w = synth.Workload("t", T, d, F, V, "fp32", "zipf")
    inp = synth.make_inputs(w, seed=81)
    states = [runner.state_from_numpy(inp, B.DTYPE_FP32, V, flags=f) for f in (0, B.FLAG_SIMT)]
    st, ref = states
    guard = torch.full((n + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    st.bufs["ws"] = guard[:n]
    B.stem_init_workspace(st.bufs["ws"])
    for s in states:
        W_up, U, dW_up = s.W_gate * 0.5, torch.empty_like(s.bufs["G"]), torch.empty_like(s.bufs["dW_gate"])
        b = s.bufs
        s.step()
        s.first = {k: b[k].clone() for k in ("y", "G", "H", "dx", "dW_gate", "dW_down", "dE_rows")}
        B.stem_dagger_forward(s.shape, s.x, s.ids, s.W_gate, W_up, s.E, s.W_down, b["y"], b["G"], b["H"], U, b["ws"])
        B.stem_dagger_backward(s.shape, s.dy, s.x, s.W_gate, W_up, s.W_down, b["G"], b["H"], U, b["perm"], b["seg_offsets"],
                               b["n_unique"], b["dx"], b["dW_gate"], dW_up, b["dW_down"], b["dE_rows"], b["ws"])
        s.first["dW_up"] = dW_up
        s.first["dagger_dx"] = b["dx"]
        assert s.status() == B.OK
    nu = int(ref.bufs["n_unique"].item())
    for k, v in ref.first.items():
        u = st.first[k]
        assert torch.equal(u[:nu], v[:nu]) if k == "dE_rows" else torch.equal(u, v), k
    assert (guard[n:] == 0x5A).all()
    # the host-buffer step in an arena of that size
    arena = torch.full((n_arena + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    B.stem_init_workspace(arena[:n_arena])
    host = {k: getattr(st, k).cpu().pin_memory() for k in ("x", "dy", "ids")}
    y, dx = (torch.zeros(T, d).pin_memory() for _ in range(2))
    cnt = torch.zeros(1, dtype=torch.int32).pin_memory()
    b = st.bufs
    B.stem_ffn_step_host(st.shape, host["x"], host["ids"], host["dy"], st.W_gate, st.E, st.W_down, y, dx, b["dW_gate"],
                         b["dW_down"], b["dE_rows"], b["unique_ids"], b["n_unique"], cnt, arena[:n_arena])
    B.stem_ffn_step_host_flush()
    torch.cuda.synchronize()
    assert B.stem_query_status(arena) == B.OK and int(cnt[0]) == nu
    assert torch.equal(y, ref.first["y"].cpu()) and torch.equal(dx, ref.first["dx"].cpu())
    assert (arena[n_arena:] == 0x5A).all()
