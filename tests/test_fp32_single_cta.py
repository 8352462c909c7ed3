"""FLAG_SINGLE_CTA reaches the fp32 contractions: they run on single CTAs, with parity, at sizes where the plan
takes pairs otherwise (several rounds of tiles, one round, a launch cut along k)."""
import re

import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import synth
from parity_measures import TOL_FP32
from test_gpu_parity import _full_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,F", [(65, 68, 132), (777, 700, 1500), (1500, 260, 2820)])
def test_layer_on_single_ctas(T, d, F):
    w = synth.Workload("t", T, d, F, 500, "fp32", "zipf")
    inp = synth.make_inputs(w, seed=34)
    ctas = {}
    for flags in (0, B.FLAG_SINGLE_CTA):
        with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as prof:
            _full_parity(w, inp, B.DTYPE_FP32, TOL_FP32, flags)
            torch.cuda.synchronize()
        names = [e.key for e in prof.key_averages() if "split_gemm_kernel" in e.key]
        ctas[flags] = {int(re.search(r"split_gemm_kernel<[^>]*, (\d)>", n).group(1)) for n in names}
    assert ctas[B.FLAG_SINGLE_CTA] == {1}, ctas
    assert T < 700 or 2 in ctas[0], ctas
