"""The work that users of this package have it do, as measurable cases.

Every case goes through the public entry points the way a program does: ``runner.LayerState``,
``runner.HostTableStack`` and the ``binding`` calls.  A case names a ``kind`` (which calls), the
layer's sizes and the types; ``prepare`` makes what the program holds before the call (weights,
table, activations, token ids, workspace), ``run`` is one pass.

Kinds, and what each stands for in use:

    forward     inference on a device-resident table: one decode step of a batch (few positions) or
                the prefill of prompts (up to one long context); nothing is kept for a backward pass
    decode_lfu  a window of decode steps of a server that keeps the table in host memory and the
                frequent rows in an on-device hot set: count the lookups, dedup, fetch the rows, forward
    train       one training step of a layer: dedup, forward, backward
    micro       a training step in two micro-batches whose weight gradients accumulate
    dagger      a training step of the STEM-dagger variant
    host_stack  a training step of several layers whose tables live in host memory: rows prefetched,
                gradient rows written back
    step_host   a training step whose batch starts and ends in pinned host buffers
"""
import math

import torch

from paper_2601_10639_b200 import binding as B
from paper_2601_10639_b200 import runner, synth

VOCAB = 32000            # vocabulary of the package's own 350M- and 1B-class workloads
LFU_STEPS = 8            # decode steps of one counting window
FP32, BF16 = "fp32", "bf16"


def _case(kind, T, d, F, ids="zipf", dtype=BF16, grad=FP32, V=VOCAB, layers=1, hot=0, **more):
    return dict(kind=kind, T=T, d_model=d, d_ff=F, V=V, ids=ids, dtype=dtype, grad=grad, layers=layers, hot=hot, **more)


def listed():
    return [
        # a decode step of a small serving batch: 16 sequences, one new token each, 1B-class layer
        _case("forward", 16, 2048, 8192, name="decode_1b_16"),
        # decode of 256 sequences, table in host memory, hot set the size of the removed up-projection
        _case("decode_lfu", 256, 2048, 8192, hot=2048, name="decode_1b_256_lfu"),
        # prefill of one prompt of an arbitrary length, 350M-class layer
        _case("forward", 1531, 1024, 2816, name="prefill_350m_1531"),
        # prefill of one long context, more distinct ids than in ordinary text, 1B-class layer
        _case("forward", 32768, 2048, 8192, ids="mix", name="prefill_1b_32k"),
        # training steps at the package's two bf16 training configurations, fp32 gradients
        _case("train", 16384, 1024, 2816, name="train_350m_16k"),
        _case("train", 16384, 2048, 8192, name="train_1b_16k"),
        # gradient accumulation with bf16 gradients: two packed micro-batches of no round length
        _case("micro", 6001, 2048, 8192, grad=BF16, name="train_1b_micro_6001"),
        # the paper's ablation that keeps the up-projection, 350M-class layer
        _case("dagger", 8192, 1024, 2816, name="dagger_350m_8k"),
        # fp32 throughout: the package's small configuration, and one sequence at 350M-class sizes
        # (what a low-precision run is checked against)
        _case("train", 256, 256, 688, ids="uniform", dtype=FP32, V=4096, name="train_fp32_256"),
        _case("train", 2048, 1024, 2816, dtype=FP32, name="train_fp32_350m_2k"),
        # tables off the device: three layers, prefetch and write-back under the layers' kernels
        _case("host_stack", 8192, 1024, 2816, layers=3, name="host_stack_350m_8k"),
        # a training step from pinned host buffers, the batch in and y, dx out over the host link
        _case("step_host", 16384, 2048, 8192, name="step_host_1b_16k"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: any kind, 350M-class to 1B-class layers and sizes between
    them that are multiples of 8 only, batches over each kind's range, either gradient type."""
    kind = rng.choice(["forward", "forward", "forward", "train", "train", "train", "train_fp32", "micro", "dagger",
                       "decode_lfu", "host_stack", "step_host"])
    d, F = rng.choice([(1024, 2816), (2048, 8192), (8 * rng.randint(96, 256), 8 * rng.randint(256, 1024))])
    grad = rng.choice([FP32, FP32, BF16])
    ids = rng.choice(["zipf", "zipf", "mix"])
    if kind == "forward":
        return _case(kind, _log_uniform(rng, 1, 32768), d, F, ids=ids)
    if kind == "decode_lfu":
        return _case(kind, _log_uniform(rng, 16, 512), d, F, hot=rng.choice([1024, 2048, 8192]))
    if kind == "train_fp32":
        return _case("train", _log_uniform(rng, 128, 2048), 4 * rng.randint(64, 256), 4 * rng.randint(160, 704),
                     ids=rng.choice(["uniform", "zipf"]), dtype=FP32, V=rng.choice([4096, VOCAB]))
    if kind == "host_stack":
        return _case(kind, _log_uniform(rng, 2048, 8192), 1024, 2816, ids=ids, grad=grad, layers=3)
    if kind == "step_host":
        return _case(kind, _log_uniform(rng, 2048, 16384), d, F, ids=ids, grad=grad)
    if kind == "dagger":
        return _case(kind, _log_uniform(rng, 512, 8192), d, F, ids=ids, grad=grad)
    return _case(kind, _log_uniform(rng, 512, 16384), d, F, ids=ids, grad=grad)


# ---- inputs ---------------------------------------------------------------------------------------
def _dtypes(case):
    return (B.DTYPE_FP32 if case["dtype"] == FP32 else B.DTYPE_BF16,
            B.DTYPE_FP32 if case["grad"] == FP32 else B.DTYPE_BF16)


def _normal(gen, shape, std, dt):
    return torch.randn(shape, generator=gen, device="cuda").mul_(std).to(dt)


def _ids(case, T, seed, layer=0):
    return torch.from_numpy(synth.token_ids(seed, T, case["V"], case["ids"], layer=layer)).cuda()


def _pinned_like(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True)


def _to_pinned(t):
    h = _pinned_like(t)
    h.copy_(t)
    return h


def _zero_partial(b):
    """Buffers of which a call writes only the first n_unique entries start from zero."""
    for k in ("unique_ids", "seg_offsets", "dE_rows"):
        if k in b:
            b[k].zero_()


def _layer(case, gen, seed, T, flags=0, backward=True, share=None):
    """A LayerState with inputs drawn as the package's workloads are: x, dy ~ N(0,1), weights
    N(0, 1/fan_in), table N(0, 0.02^2)."""
    code, grad = _dtypes(case)
    dt = runner.torch_dtype(code)
    d, F, V = case["d_model"], case["d_ff"], case["V"]
    st = runner.LayerState(B.make_shape(T, d, F, V, code, grad, flags))
    st.x = _normal(gen, (T, d), 1.0, dt)
    st.ids = _ids(case, T, seed)
    if backward:
        st.dy = _normal(gen, (T, d), 1.0, dt)
    if share is None:
        st.W_gate = _normal(gen, (F, d), d ** -0.5, dt)
        st.W_down = _normal(gen, (d, F), F ** -0.5, dt)
        st.E = _normal(gen, (V, F), 0.02, dt)
    else:
        st.W_gate, st.W_down, st.E = share.W_gate, share.W_down, share.E
    st.allocate(backward)
    _zero_partial(st.bufs)
    return st


def _outputs(b, names):
    return {k: b[k] for k in names}


INDEX = ("unique_ids", "n_unique", "inverse", "perm", "seg_offsets")
GRADS = ("dx", "dW_gate", "dW_down", "dE_rows")


# ---- one preparation and one pass per kind ----------------------------------------------------------
def _prepare_layer(case, gen, seed):
    """forward and train."""
    backward = case["kind"] == "train"
    st = _layer(case, gen, seed, case["T"], backward=backward)
    return {"st": st, "backward": backward}


def _run_layer(s):
    st = s["st"]
    if not s["backward"]:
        st.forward(save=False)
        return st.bufs["y"]
    st.step()
    return _outputs(st.bufs, ("y", "G", "H") + INDEX + GRADS)


def _prepare_micro(case, gen, seed):
    T1 = case["T"] // 2
    first = _layer(case, gen, seed, T1)
    second = _layer(case, gen, seed + 1000003, case["T"] - T1, flags=B.FLAG_ACCUM_GRADS, share=first)
    for k in ("dW_gate", "dW_down"):
        second.bufs[k] = first.bufs[k]
    return {"parts": [first, second]}


def _run_micro(s):
    for st in s["parts"]:
        st.step()
    return [_outputs(st.bufs, ("y",) + INDEX + GRADS) for st in s["parts"]]


def _prepare_dagger(case, gen, seed):
    st = _layer(case, gen, seed, case["T"])
    T, d, F = case["T"], case["d_model"], case["d_ff"]
    W_up = _normal(gen, (F, d), d ** -0.5, st.x.dtype)
    st.bufs["U"] = torch.empty(T, F, dtype=st.x.dtype, device="cuda")
    st.bufs["dW_up"] = torch.empty_like(st.bufs["dW_gate"])
    return {"st": st, "W_up": W_up}


def _run_dagger(s):
    st, W_up, b = s["st"], s["W_up"], s["st"].bufs
    st.dedup()
    B.stem_dagger_forward(st.shape, st.x, st.ids, st.W_gate, W_up, st.E, st.W_down, b["y"], b["G"], b["H"], b["U"], b["ws"])
    B.stem_dagger_backward(st.shape, st.dy, st.x, st.W_gate, W_up, st.W_down, b["G"], b["H"], b["U"], b["perm"],
                           b["seg_offsets"], b["n_unique"], b["dx"], b["dW_gate"], b["dW_up"], b["dW_down"], b["dE_rows"],
                           b["ws"])
    return _outputs(b, ("y", "G", "H", "U", "dW_up") + INDEX + GRADS)


def _prepare_decode_lfu(case, gen, seed):
    st = _layer(case, gen, seed, case["T"], backward=False)
    table = _to_pinned(st.E)
    # the Zipfian ids are ranked by frequency, so the hot set of a warm cache holds the smallest ones
    hot_rows, hot_slot = runner.build_hot_set(table, torch.arange(case["hot"]))
    st.E = None
    T, d, F, V = case["T"], case["d_model"], case["d_ff"], case["V"]
    R = min(T, V)
    code, grad = _dtypes(case)
    return {
        "st": st, "table": table, "hot_rows": hot_rows, "hot_slot": hot_slot,
        "freq": torch.zeros(V, dtype=torch.int32, device="cuda"),
        "hits": torch.zeros(2, dtype=torch.int32, device="cuda"),
        "rows": torch.zeros(2, dtype=torch.int32, device="cuda"),
        "cache": torch.zeros(R, F, dtype=st.x.dtype, device="cuda"),
        "cache_shape": B.make_shape(T, d, F, R, code, grad, 0),
        "ids": [_ids(case, T, seed, layer=1 + i) for i in range(LFU_STEPS)],
        "x": [_normal(gen, (T, d), 1.0, st.x.dtype) for _ in range(LFU_STEPS)],
        "y": [torch.empty(T, d, dtype=st.x.dtype, device="cuda") for _ in range(LFU_STEPS)],
    }


def _run_decode_lfu(s):
    st, b = s["st"], s["st"].bufs
    for k in ("freq", "hits", "rows"):      # a counting window begins
        s[k].zero_()
    for ids, x, y in zip(s["ids"], s["x"], s["y"]):
        B.stem_lfu_touch(st.shape.T, st.shape.V, ids, s["freq"], s["hot_slot"], s["hits"])
        B.stem_dedup_ids(st.shape, ids, b["unique_ids"], b["n_unique"], b["inverse"], b["perm"], b["seg_offsets"], b["ws"])
        B.stem_prefetch_rows_hot(st.shape, b["unique_ids"], b["n_unique"], s["table"], s["hot_rows"], s["hot_slot"],
                                 s["cache"], s["rows"], b["ws"])
        B.stem_ffn_forward(s["cache_shape"], x, b["inverse"], st.W_gate, s["cache"], st.W_down, y, None, None, b["ws"])
    # y holds every step's rows; the index arrays of a step are scratch of its forward
    return {"y": s["y"], "freq": s["freq"], "hits": s["hits"], "rows": s["rows"]}


def _prepare_host_stack(case, gen, seed):
    code, grad = _dtypes(case)
    dt, gdt = runner.torch_dtype(code), runner.torch_dtype(grad)
    T, d, F, V, L = case["T"], case["d_model"], case["d_ff"], case["V"], case["layers"]
    W_gate = _normal(gen, (F, d), d ** -0.5, dt)
    W_down = _normal(gen, (d, F), F ** -0.5, dt)
    tables = [_to_pinned(_normal(gen, (V, F), 0.02, dt)) for _ in range(L)]
    stack = runner.HostTableStack(B.make_shape(T, d, F, V, code, grad, 0), L, tables, W_gate, W_down, False)
    for k in stack.slots:
        _zero_partial(k)
        k["host_rows"].zero_()
        k["host_ids"].zero_()
    kept = [{"y": torch.empty(T, d, dtype=dt, device="cuda"), "dx": torch.empty(T, d, dtype=dt, device="cuda"),
             "dW_gate": torch.empty(F, d, dtype=gdt, device="cuda"), "dW_down": torch.empty(d, F, dtype=gdt, device="cuda")}
            for _ in range(L)]
    return {
        "stack": stack, "kept": kept,
        "x": [_normal(gen, (T, d), 1.0, dt) for _ in range(L)],
        "dy": [_normal(gen, (T, d), 1.0, dt) for _ in range(L)],
        "ids": [_ids(case, T, seed, layer=i) for i in range(L)],
    }


def _run_host_stack(s):
    stack, kept = s["stack"], s["kept"]

    def keep(l, slot):      # the layers are independent: each one's results leave the shared buffers
        for k, v in kept[l].items():
            v.copy_(getattr(stack, k))

    stack.step(s["x"], s["ids"], s["dy"], keep)
    stack.finish()
    return {"layers": kept, "host": [_outputs(k, ("host_rows", "host_ids", "host_n")) for k in stack.slots]}


def _prepare_step_host(case, gen, seed):
    st = _layer(case, gen, seed, case["T"])
    host = {k: _to_pinned(getattr(st, k)) for k in ("x", "ids", "dy")}
    host.update(y=_pinned_like(st.x), dx=_pinned_like(st.x), n=torch.zeros(1, dtype=torch.int32, pin_memory=True))
    b = st.bufs
    s = {"shape": st.shape, "W_gate": st.W_gate, "W_down": st.W_down, "E": st.E, "host": host,
         **{k: b[k] for k in ("dW_gate", "dW_down", "dE_rows", "unique_ids", "n_unique")}}
    del st, b
    s["arena"] = torch.empty(B.stem_step_arena_bytes(s["shape"]), dtype=torch.uint8, device="cuda")
    B.stem_init_workspace(s["arena"])
    return s


def _run_step_host(s):
    h = s["host"]
    B.stem_ffn_step_host(s["shape"], h["x"], h["ids"], h["dy"], s["W_gate"], s["E"], s["W_down"], h["y"], h["dx"],
                         s["dW_gate"], s["dW_down"], s["dE_rows"], s["unique_ids"], s["n_unique"], h["n"], s["arena"])
    B.stem_ffn_step_host_flush()
    return {**_outputs(h, ("y", "dx", "n")), **_outputs(s, ("dW_gate", "dW_down", "dE_rows", "unique_ids"))}


_KINDS = {
    "forward": (_prepare_layer, _run_layer),
    "train": (_prepare_layer, _run_layer),
    "micro": (_prepare_micro, _run_micro),
    "dagger": (_prepare_dagger, _run_dagger),
    "decode_lfu": (_prepare_decode_lfu, _run_decode_lfu),
    "host_stack": (_prepare_host_stack, _run_host_stack),
    "step_host": (_prepare_step_host, _run_step_host),
}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    state = _KINDS[case["kind"]][0](case, gen, seed)
    state["kind"] = case["kind"]
    return state


def run(state):
    return _KINDS[state["kind"]][1](state)


# ---- what a pass cannot do without -------------------------------------------------------------------
def _distinct(case, T):
    """About how many distinct ids T positions have (each one's table row is read once)."""
    V = case["V"]
    ids = synth.token_ids(synth.BASE_SEED, min(T, 65536), V, case["ids"])
    return len(set(ids.tolist()))


def _work_layer(case, T, backward, saved, contractions):
    """One layer on T positions: weights, activations and the table rows of its distinct ids read
    once, every output written once; 2 T d F floating-point operations per contraction."""
    d, F = case["d_model"], case["d_ff"]
    e = 4 if case["dtype"] == FP32 else 2
    g = 4 if case["grad"] == FP32 else 2
    n = _distinct(case, T)
    byts = T * d * e + 4 * T + 2 * d * F * e + n * F * e + T * d * e          # x, ids, weights, rows; y
    if saved:
        byts += 2 * T * F * e                                                 # G, H
    if backward:
        byts += T * d * e + T * d * e + 2 * d * F * g + n * F * g             # dy; dx, dW, dE rows
        byts += 4 * (3 * T + 2 * n)                                           # index arrays
    return byts, 2.0 * T * d * F * contractions


def work(case):
    kind, T = case["kind"], case["T"]
    d, F = case["d_model"], case["d_ff"]
    if kind == "forward":
        b, f = _work_layer(case, T, False, False, 2)
    elif kind == "decode_lfu":
        b, f = _work_layer(case, T, False, False, 2)
        b, f = b * LFU_STEPS, f * LFU_STEPS                                   # the weights again in every step
    elif kind == "train":
        b, f = _work_layer(case, T, True, True, 6)
    elif kind == "micro":
        T1 = T // 2
        b1, f1 = _work_layer(case, T1, True, True, 6)
        b2, f2 = _work_layer(case, T - T1, True, True, 6)
        b, f = b1 + b2, f1 + f2
    elif kind == "dagger":
        b, f = _work_layer(case, T, True, True, 9)
        b += T * F * 2 + d * F * (2 + (4 if case["grad"] == FP32 else 2))     # U; W_up, dW_up
    elif kind == "host_stack":
        b, f = _work_layer(case, T, True, True, 6)
        b += _distinct(case, T) * F * (2 + (4 if case["grad"] == FP32 else 2))  # rows in, gradient rows out
        b, f = b * case["layers"], f * case["layers"]
    else:
        b, f = _work_layer(case, T, True, True, 6)
        b += 4 * T * d * 2                                                    # x, dy in; y, dx out
    return {"bytes": float(b), "flops": f}


def tolerance(case):
    """About four times what the path differs from the same formulas in 64 bits.  fp32: up to 1.2e-6
    of the norm, 8e-6 of a value (5e-5 in table-gradient rows).  bf16: 2.4e-3 and 1e-2 forward, 3.3e-3
    and 2e-2 in the gradients; a table-gradient row can be a sum of large terms that cancel, where the
    bf16 rounding of the terms is up to 0.26 of the output's root mean square."""
    if case["dtype"] == FP32:
        return {"rel": 5e-6, "max": 2e-4}
    if case["kind"] in ("forward", "decode_lfu"):
        return {"rel": 1e-2, "max": 0.04}
    return {"rel": 1.3e-2, "max": 0.9}


# ---- the same outputs in 64 bits, in plain torch ------------------------------------------------------
def _pad_rows(t, rows):
    out = torch.zeros((rows,) + tuple(t.shape[1:]), dtype=t.dtype, device=t.device)
    out[:t.shape[0]] = t
    return out


def _exact_layer(x, ids, dy, W_gate, W_down, E, W_up=None):
    """The layer's formulas in fp64 (dy None: the forward alone); table-gradient rows of the distinct
    ids in ascending order."""
    ids = ids.long()
    x, Wg, Wd = x.double(), W_gate.double(), W_down.double()
    u = E[ids].double()
    if W_up is not None:
        u = u + x @ W_up.double().T
    g = x @ Wg.T
    s = torch.sigmoid(g)
    h = g * s * u
    o = {"y": h @ Wd.T}
    if dy is None:
        return o
    dy = dy.double()
    o.update(G=g, H=h, U=u)
    dh = dy @ Wd
    o["dW_down"] = dy.T @ h
    du = dh * (g * s)
    dg = dh * u * (s * (1 + g * (1 - s)))
    o["dx"] = dg @ Wg
    o["dW_gate"] = dg.T @ x
    if W_up is not None:
        o["dx"] = o["dx"] + du @ W_up.double()
        o["dW_up"] = du.T @ x
    unique, inverse = torch.unique(ids, return_inverse=True)
    o["dE_rows"] = torch.zeros(unique.numel(), E.shape[1], dtype=torch.float64, device=u.device).index_add_(0, inverse, du)
    return o


def _exact_state(st, more=(), W_up=None):
    e = _exact_layer(st.x, st.ids, st.dy, st.W_gate, st.W_down, st.E, W_up)
    e["dE_rows"] = _pad_rows(e["dE_rows"], st.bufs["dE_rows"].shape[0])
    out = {k: e[k] for k in ("y",) + tuple(more) + GRADS}
    out.update({k: None for k in INDEX})         # whole numbers: either side has the one right value
    return out


def exact(case, seed):
    """What `run` returns for these inputs, in 64 bits (None for the index arrays and counters)."""
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "forward":
        st = s["st"]
        return _exact_layer(st.x, st.ids, None, st.W_gate, st.W_down, st.E)["y"]
    if kind == "train":
        return _exact_state(s["st"], ("G", "H"))
    if kind == "micro":
        parts = [_exact_state(st) for st in s["parts"]]
        for k in ("dW_gate", "dW_down"):         # both micro-batches add to the same buffers
            parts[0][k] = parts[1][k] = parts[0][k] + parts[1][k]
        return parts
    if kind == "dagger":
        return _exact_state(s["st"], ("G", "H", "U", "dW_up"), s["W_up"])
    if kind == "decode_lfu":
        st, table = s["st"], s["table"].cuda()
        y = [_exact_layer(x, ids, None, st.W_gate, st.W_down, table)["y"] for ids, x in zip(s["ids"], s["x"])]
        return {"y": y, "freq": None, "hits": None, "rows": None}
    if kind == "host_stack":
        stack = s["stack"]
        layers, host = [], []
        for i in range(case["layers"]):
            e = _exact_layer(s["x"][i], s["ids"][i], s["dy"][i], stack.W_gate, stack.W_down, stack.tables[i].cuda())
            layers.append({k: e[k] for k in ("y", "dx", "dW_gate", "dW_down")})
            host.append({"host_rows": _pad_rows(e["dE_rows"], stack.R), "host_ids": None, "host_n": None})
        return {"layers": layers, "host": host}
    h = {k: s["host"][k].cuda() for k in ("x", "ids", "dy")}
    e = _exact_layer(h["x"], h["ids"], h["dy"], s["W_gate"], s["W_down"], s["E"])
    out = {k: e[k] for k in ("y", "dx", "dW_gate", "dW_down")}
    out.update(dE_rows=_pad_rows(e["dE_rows"], s["dE_rows"].shape[0]), n=None, unique_ids=None)
    return out
