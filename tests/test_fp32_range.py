"""fp32 contractions whose two operands are of very different magnitude, down to subnormal numbers, in all three
operand layouts, and with values that the three bf16 parts do not carry, against the chain of FMAs in fp32
(FLAG_SIMT)."""
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


def _spoiled(T, d, F, where, flags):
    """A layer with one operand value that the parts do not carry, or (`edge`) the largest that they do."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(72)
    st = runner.LayerState(B.make_shape(T, d, F, 90, B.DTYPE_FP32, B.DTYPE_FP32, flags))
    st.x, st.dy = (torch.randn(T, d, generator=gen, device="cuda") for _ in range(2))
    st.W_gate = torch.randn(F, d, generator=gen, device="cuda") * d ** -0.5
    st.W_down = torch.randn(d, F, generator=gen, device="cuda") * F ** -0.5
    st.E = torch.randn(90, F, generator=gen, device="cuda")
    st.ids = torch.randint(0, 90, (T,), generator=gen, device="cuda", dtype=torch.int32)
    st.W_up = torch.randn(F, d, generator=gen, device="cuda") * d ** -0.5
    st.allocate()
    for k in ("dW_gate", "dW_down"):
        st.bufs[k].normal_(generator=gen)
    st.bufs["U"], st.bufs["dW_up"] = torch.empty_like(st.bufs["G"]), torch.zeros_like(st.bufs["dW_gate"])
    at = {"dy_inf": (st.dy, (T - 1, d - 1), float("inf")), "x_nan": (st.x, (T // 2, 0), float("nan")),
          "w_large": (st.W_gate, (F - 1, d // 2), 3.4e38), "x_2^24": (st.x, (0, d - 1), 2.0 ** 24),
          "w_down_inf": (st.W_down, (0, F - 1), -float("inf"))}
    t, i, v = at[where]
    t[i] = v
    return st


OUTPUTS = ("y", "G", "H", "dx", "dW_gate", "dW_down", "dE_rows")


@pytest.mark.parametrize("where", ["dy_inf", "x_nan", "w_large", "x_2^24", "w_down_inf"])
@pytest.mark.parametrize("T,d,F,flags", [(1, 8, 12, 0), (70, 260, 332, B.FLAG_ACCUM_GRADS), (4099, 136, 268, 0), (1500, 516, 1024, 0)])
def test_values_beyond_the_parts(T, d, F, flags, where):
    """The launches that meet them give what the FMA kernels give, in a time like theirs."""
    out, times = [], []
    for f in (flags, flags | B.FLAG_SIMT):
        st = _spoiled(T, d, F, where, f)
        st.step()
        assert st.status() == B.OK
        out.append({k: st.bufs[k].clone() for k in OUTPUTS})
        n = int(st.bufs["n_unique"].item())
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ev[0].record()
        st.backward()
        ev[1].record()
        torch.cuda.synchronize()
        times.append(ev[0].elapsed_time(ev[1]))
    a, b = out
    for k in OUTPUTS:
        u, v = (o[k][:n] if k == "dE_rows" else o[k] for o in (a, b))
        if where == "dy_inf" and k in ("y", "G", "H"):      # no such value in the forward pass: the parts carry it
            assert (u - v).norm() <= 4e-6 * v.norm(), k
        else:
            # A contraction of ordinary operands in the same pass (or one fed by such a one) differs by its rounding
            bad = ~torch.isfinite(v)
            assert torch.equal(u[bad].nan_to_num(), v[bad].nan_to_num()) and torch.equal(u.isnan(), v.isnan()), k
            u, v = u[~bad], v[~bad]
            assert torch.equal(u, v) or (u - v).abs().max() <= 1e-5 * v.abs().max(), k
    assert times[0] <= 4 * times[1] + 0.2, times          # (a chain per result took hundreds of times as long)


@pytest.mark.parametrize("where", ["dy_inf", "x_nan", "w_down_inf"])
def test_values_beyond_the_parts_dagger(where):
    out = []
    for flags in (0, B.FLAG_SIMT):
        st = _spoiled(333, 132, 260, where, flags)
        b = st.bufs
        st.dedup()
        B.stem_dagger_forward(st.shape, st.x, st.ids, st.W_gate, st.W_up, st.E, st.W_down, b["y"], b["G"], b["H"], b["U"], b["ws"])
        B.stem_dagger_backward(st.shape, st.dy, st.x, st.W_gate, st.W_up, st.W_down, b["G"], b["H"], b["U"], b["perm"],
                               b["seg_offsets"], b["n_unique"], b["dx"], b["dW_gate"], b["dW_up"], b["dW_down"], b["dE_rows"], b["ws"])
        assert st.status() == B.OK
        n = int(b["n_unique"].item())
        out.append({k: b[k][:n] if k == "dE_rows" else b[k] for k in OUTPUTS + ("U", "dW_up")})
    for k, v in out[1].items():
        u = out[0][k]
        bad = ~torch.isfinite(v)
        assert torch.equal(u.isnan(), v.isnan()) and torch.equal(u[bad].nan_to_num(), v[bad].nan_to_num()), k
        if not bad.all():
            assert (u[~bad] - v[~bad]).abs().max() <= 1e-5 * v[~bad].abs().max(), k
