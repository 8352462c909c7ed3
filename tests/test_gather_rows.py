"""Row gathers from a host table on both sides of the sizes where the launch changes, with and without a hot set: the
rows, the counts, and how many CTAs the launch takes (a plain gather shares the SMs with another layer's kernels)."""
import json

import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner

pytestmark = pytest.mark.gpu


def _table(V, F):
    gen = torch.Generator()
    gen.manual_seed(91)
    return torch.randint(-2 ** 15, 2 ** 15, (V, F), generator=gen, dtype=torch.int16).pin_memory()


@pytest.mark.parametrize("F", [8, 136, 2816])
@pytest.mark.parametrize("T", [1, 255, 511, 512, 513, 1023, 1024, 1025, 1300])
@pytest.mark.parametrize("hot", [0, 400])
def test_rows(T, F, hot):
    V = 1500
    table = _table(V, F)
    shape = B.make_shape(T, 8, F, V, B.DTYPE_BF16, B.DTYPE_FP32, 0)
    ws = torch.empty(B.stem_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    B.stem_init_workspace(ws)
    if hot:
        hot_rows, hot_slot = runner.build_hot_set(table, torch.arange(0, V, 3)[:hot])
    for n in {T, T // 2 + 1}:
        gen = torch.Generator()
        gen.manual_seed(T + n)
        ids = torch.randperm(V, generator=gen)[:T].int()
        out = torch.full((T, F), 77, dtype=torch.int16, device="cuda")
        n_ids = torch.tensor([n], dtype=torch.int32, device="cuda")
        stats = torch.zeros(2, dtype=torch.int32, device="cuda")
        if hot:
            B.stem_prefetch_rows_hot(shape, ids.cuda(), n_ids, table, hot_rows, hot_slot, out, stats, ws)
        else:
            B.stem_prefetch_rows(shape, ids.cuda(), n_ids, table, out, ws)
        assert B.stem_query_status(ws) == B.OK
        assert torch.equal(out[:n].cpu(), table[ids[:n].long()]) and (out[n:] == 77).all()
        if hot:
            hits = int((hot_slot.cpu()[ids[:n].long()] >= 0).sum())
            assert stats.tolist() == [hits, n - hits]


def _ctas(T, F, hot, tmp_path):
    V = 4000
    table = torch.zeros(V, F, dtype=torch.bfloat16).pin_memory()
    shape = B.make_shape(T, 8, F, V, B.DTYPE_BF16, B.DTYPE_FP32, 0)
    ws = torch.empty(B.stem_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    B.stem_init_workspace(ws)
    ids = torch.arange(T, device="cuda", dtype=torch.int32)
    n_ids = torch.tensor([T], dtype=torch.int32, device="cuda")
    out = torch.empty(T, F, dtype=torch.bfloat16, device="cuda")
    hot_rows, hot_slot = runner.build_hot_set(table, torch.arange(100))
    with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as prof:
        if hot:
            B.stem_prefetch_rows_hot(shape, ids, n_ids, table, hot_rows, hot_slot, out, None, ws)
        else:
            B.stem_prefetch_rows(shape, ids, n_ids, table, out, ws)
        torch.cuda.synchronize()
    path = str(tmp_path / "trace.json")
    prof.export_chrome_trace(path)
    events = [e for e in json.load(open(path))["traceEvents"] if "gather_rows_kernel" in str(e.get("name")) and "grid" in e.get("args", {})]
    assert len(events) == 1
    return events[0]["args"]["grid"][0]


@pytest.mark.parametrize("T,F,hot,ctas", [
    (256, 8192, False, 32), (512, 8192, False, 32), (513, 8192, False, 64), (300, 5120, False, 51),
    (256, 2816, False, 64), (20, 2816, False, 20), (2048, 2816, False, 64),
    (200, 8192, True, 200), (512, 8192, True, 512), (1024, 2816, True, 512), (1025, 2816, True, 64),
])
def test_ctas(T, F, hot, ctas, tmp_path):
    assert _ctas(T, F, hot, tmp_path) == ctas
