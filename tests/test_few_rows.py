"""bf16 layers on few rows (decode steps, short prompts) vs the CPU checker: the weight-streaming kernels at
the edges of their padding (16 and 32 rows), of the batch they take, of W's 128-row tiles and 64-wide k blocks
(one block, fewer blocks than a cluster has CTAs, a ragged last one), and the half-width tiles of the general kernel."""
import numpy as np
import pytest
import torch

from oracle import stem_oracle as O
from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth
from parity_measures import TOL_BF16, assert_close
from test_gpu_parity import _full_parity, _np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,F", [
    (1, 8, 8), (1, 2048, 2056), (15, 264, 520), (16, 1024, 2816), (17, 136, 4104), (32, 72, 1032), (33, 1032, 264),
    (64, 64, 9000), (97, 520, 1160), (128, 1024, 2816), (129, 1024, 2816), (200, 264, 2568), (256, 136, 5000),
])
def test_forward_few_rows(T, d, F):
    w = synth.Workload("t", T, d, F, 300, "bf16", "zipf")
    inp = synth.make_inputs(w, seed=41)
    st = runner.state_from_numpy(inp, B.DTYPE_BF16, w.V, backward=False)
    st.forward()
    assert st.status() == B.OK
    y_ref, im = O.forward(inp["x"], inp["ids"], inp["W_gate"], inp["E"], inp["W_down"], True)
    for k, ref in (("G", im["G"]), ("H", im["H"]), ("y", y_ref)):
        assert_close(_np(st.bufs[k]), ref, TOL_BF16, k)
    y = st.bufs["y"].clone()
    st.bufs["y"].fill_(float("nan"))
    st.forward(save=False)                       # H in the workspace, G nowhere
    assert st.status() == B.OK and torch.equal(st.bufs["y"], y)


@pytest.mark.parametrize("T,d,F", [(300, 264, 520), (700, 1024, 2816)])
def test_layer_half_width_tiles(T, d, F):
    w = synth.Workload("t", T, d, F, 300, "bf16", "zipf")
    _full_parity(w, synth.make_inputs(w, seed=43), B.DTYPE_BF16, TOL_BF16)


def test_few_rows_bad_id_is_clamped_and_reported():
    w = synth.Workload("t", 20, 136, 264, 50, "bf16", "uniform")
    inp = synth.make_inputs(w, seed=42)
    st = runner.state_from_numpy(inp, B.DTYPE_BF16, w.V, backward=False)
    good = np.clip(inp["ids"], 1, 48)
    bad = good.copy()
    good[3], good[11] = 49, 0
    bad[3], bad[11] = 50, -7
    out = []
    for ids in (good, bad):
        st.ids = torch.from_numpy(ids).cuda()
        st.forward()
        out.append(st.bufs["y"].clone())
    assert torch.equal(out[0], out[1])
    assert st.status() == B.ERR_ID_RANGE
