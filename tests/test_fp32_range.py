"""fp32 contractions whose two operands are of very different magnitude, down to subnormal numbers, in all three
operand layouts, against the chain of FMAs in fp32 (FLAG_SIMT)."""
import pytest
import torch

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner

pytestmark = pytest.mark.gpu


def _state(T, d, F, V, small, large, flags):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(71)

    def normal(shape, scale):
        return (torch.randn(shape, generator=gen, device="cuda").double() * scale).float()

    st = runner.LayerState(B.make_shape(T, d, F, V, B.DTYPE_FP32, B.DTYPE_FP32, flags))
    st.x, st.dy = normal((T, d), small), normal((T, d), small)
    st.W_gate, st.W_down, st.E = normal((F, d), large), normal((d, F), large), normal((V, F), 1.0 / large)
    st.ids = torch.randint(0, V, (T,), generator=gen, device="cuda", dtype=torch.int32)
    st.allocate()
    st.dedup()
    saved = normal((T, F), 1.0), normal((T, F), large), normal((T, d), large)
    return st, saved


# (the last two stay inside what the parts carry; the first three have partners of any size)
@pytest.mark.parametrize("small,large", [(1e-36, 1e8), (1e-38, 1e10), (1e-41, 1e12), (1e-36, 1e6), (1e-41, 1e5)])
@pytest.mark.parametrize("T,d,F", [(70, 260, 332), (300, 256, 688)])
def test_small_against_large(T, d, F, small, large):
    """Forward: x (small) W_gate (large), then H (small) W_down (large).  Backward, on saved G and H of its own:
    dy (small) W_down (large), dG (small) W_gate (large), dy^T H and dG^T x (small by large, over the positions)."""
    out = []
    for flags in (0, B.FLAG_SIMT):
        st, (G, H, x) = _state(T, d, F, 60, small, large, flags)
        st.forward()
        got = {k: st.bufs[k].double() for k in ("G", "H", "y")}
        st.bufs["G"], st.bufs["H"], st.x = G, H, x
        st.backward()
        assert st.status() == B.OK
        got.update((k, st.bufs[k].double()) for k in ("dx", "dW_gate", "dW_down"))
        got["G_exact"] = _state(T, d, F, 60, small, large, flags)[0].x.double() @ st.W_gate.double().T
        got["dW_down_exact"] = st.dy.double().T @ H.double()
        out.append(got)
    a, b = out
    # Chains of at most 688 additions round to sqrt(688) 2^-24 = 1.6e-6 of a sum each; the operands H and dG, of the size of
    # `small` times 16, are themselves rounded to multiples of 2^-149 (at 1e-41: 1e-5 of them), not always the same way
    tol = 4e-6 + 2.0 ** -149 / (8 * small)
    for k in ("G", "H", "y", "dx", "dW_gate", "dW_down"):
        assert torch.isfinite(a[k]).all() and b[k].norm() > 0, k
        assert (a[k] - b[k]).norm() <= tol * b[k].norm(), k
    for k in ("G", "dW_down"):      # inputs as they are on both sides: 64 bits
        ref = a[k + "_exact"]
        quantum = 2.0 ** -149 * ref.numel() ** 0.5
        assert (a[k] - ref).norm() <= 2e-6 * ref.norm() + quantum, k
