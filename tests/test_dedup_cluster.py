"""Dedup in one launch of a cluster, at the edges of its range, of a CTA's chunk and of a warp's run, for one to
four radix passes; every output has one right value."""
import numpy as np
import pytest
import torch

from oracle import stem_oracle as O
from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [256, 257, 511, 1023, 1025, 1056, 4095, 8192, 8193, 16383, 16384, 16385])
@pytest.mark.parametrize("V,dist", [(200, "uniform"), (32000, "zipf"), (70001, "mix"), (1 << 26, "uniform"), (9, "same")])
def test_dedup(T, V, dist):
    ids = synth.token_ids(T + V % 97, T, V, dist)
    if T == 8193:
        ids = ids.copy()
        ids[5], ids[8192] = -3, V          # clamped to 0 and V - 1, reported
    st = runner.LayerState(B.make_shape(T, 8, 8, V, B.DTYPE_BF16, B.DTYPE_FP32, 0)).allocate(backward=False)
    st.ids = torch.from_numpy(ids).cuda()
    for _ in range(2):
        st.dedup()
        assert st.status() == (B.ERR_ID_RANGE if T == 8193 else B.OK)
        ref = O.dedup(np.clip(ids, 0, V - 1))
        n = ref["n_unique"]
        assert int(st.bufs["n_unique"].item()) == n
        for k, m in (("unique_ids", n), ("perm", T), ("inverse", T), ("seg_offsets", n + 1)):
            assert np.array_equal(st.bufs[k][:m].cpu().numpy(), ref[k]), k
