"""STEM-dagger backward on the tensor cores vs the CPU checker, where its launches can go wrong: the three weight
gradients in one launch (tiles of three products, a split last round), dx as one contraction over two pairs of
operands whose ragged 64-wide blocks do not line up (whole, and cut along k), gradients left out, gradients accumulated."""
import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from oracle import stem_oracle as O
from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth
from parity_measures import TOL_BF16, assert_close
from test_gpu_parity import _np

pytestmark = pytest.mark.gpu


def _run(T, d, F, flags, left_out=(), start=None):
    w = synth.Workload("t", T, d, F, 200, "bf16", "zipf")
    inp = synth.make_inputs(w, seed=51)
    rng = np.random.default_rng(52)
    W_up = synth.round_bf16((rng.normal(size=(F, d)) * d ** -0.5).astype(np.float32))
    st = runner.state_from_numpy(inp, B.DTYPE_BF16, w.V, flags=flags)
    dW = torch.from_numpy(W_up).cuda().bfloat16()
    b = st.bufs
    b["U"] = torch.empty(T, F, dtype=torch.bfloat16, device="cuda")
    b["dW_up"] = torch.empty_like(b["dW_gate"])
    for k in ("dW_gate", "dW_up", "dW_down"):
        b[k].fill_(0.0 if start is None else start)
    st.dedup()
    B.stem_dagger_forward(st.shape, st.x, st.ids, st.W_gate, dW, st.E, st.W_down, b["y"], b["G"], b["H"], b["U"], b["ws"])
    out = {k: (None if k in left_out else b[k]) for k in ("dx", "dW_gate", "dW_up", "dW_down", "dE_rows")}
    B.stem_dagger_backward(st.shape, st.dy, st.x, st.W_gate, dW, st.W_down, b["G"], b["H"], b["U"], b["perm"],
                           b["seg_offsets"], b["n_unique"], out["dx"], out["dW_gate"], out["dW_up"], out["dW_down"],
                           out["dE_rows"], b["ws"])
    assert st.status() == B.OK
    n = int(b["n_unique"].item())
    return inp, W_up, {k: v[:n] if k == "dE_rows" else v for k, v in out.items() if v is not None}


@pytest.mark.parametrize("flags", [0, B.FLAG_SINGLE_CTA], ids=["pair", "single"])
# splits: launches whose last round is cut along k (and then finished by tail_fixup_kernel): the weight gradients of the
# last but one size (few tiles, 8200 positions), dx of the last one (few tiles, 2 x 4104 deep, pieces on both
# sides of the change of operands); the others save too little by it
@pytest.mark.parametrize("T,d,F,splits", [(130, 72, 136, 0), (300, 264, 520, 0), (8200, 520, 1096, 0), (8200, 264, 520, 1),
                                          (300, 264, 4104, 1)])
def test_gradients(T, d, F, splits, flags):
    with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as prof:
        inp, W_up, got = _run(T, d, F, flags)
        torch.cuda.synchronize()
    ran = {e.key: e.count for e in prof.key_averages()}
    assert sum(n for k, n in ran.items() if "tc_gemm_kernel" in k) == 6      # up, gate, down; dH, three gradients, dx
    assert sum(n for k, n in ran.items() if "tail_fixup_kernel" in k) == splits, ran
    ref = O.dagger_backward(inp["dy"], inp["x"], inp["ids"], inp["W_gate"], W_up, inp["E"], inp["W_down"])
    for k in ("dx", "dW_gate", "dW_up", "dW_down", "dE_rows"):
        # a sum of few bf16-rounded terms can cancel to an entry far below them: the whole-tensor measures
        assert O.scaled_max_err(_np(got[k]), ref[k]) <= TOL_BF16 and O.rel_frobenius_err(_np(got[k]), ref[k]) <= 1e-2, k


def test_left_out_and_accumulated_gradients_agree_with_the_whole_call():
    T, d, F = 300, 264, 520
    _, _, whole = _run(T, d, F, 0)
    for left_out in (("dW_up",), ("dW_down", "dx"), ("dW_gate", "dE_rows")):
        _, _, part = _run(T, d, F, 0, left_out)
        for k, v in part.items():
            assert torch.equal(v, whole[k]), (left_out, k)
    _, _, acc = _run(T, d, F, B.FLAG_ACCUM_GRADS, start=0.5)
    for k in ("dW_gate", "dW_up", "dW_down"):
        assert (acc[k] - 0.5 - whole[k]).abs().max() <= 2e-6 * (0.5 + whole[k].abs().max()), k   # one fp32 addition
