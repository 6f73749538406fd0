"""The work that a program built on this framework has it do, as cases that can be timed and compared.

A case is one of four kinds of pass through the public entry points:

* ``linear``     one layer on its own (``linear_ex``);
* ``layer``      the seven linears of a decoder layer in the order in which a model runs them: q, k, v share one
                 activation and go out together, then o, then gate and up together, then down.  Each group reads what
                 the code between the linears (attention, norms, the activation function) left, so the groups are
                 separate calls;
* ``stack``      the linears of several decoder layers as one batch of independent calls (``linear_batched_ex``), the form
                 in which bench.py runs the full stack;
* ``calibrate``  the preparation of one layer from its weight and calibration activations
                 (``prepare_from_calibration``): W_q, the rank-k factors, quantised and packed.

Shapes are those of bench.py and of the test configurations: hidden 4096 / feed-forward 11008, hidden 5120 /
feed-forward 13824, the tiny 256 x 256 layer, ranks up to 256, 1 to 4096 tokens, fp32, bf16 and MXINT8 activations, 4- and
2-bit weights, and sizes that are no multiple of any tile.
"""
from __future__ import annotations

import torch

import paper_2402_02446_b200 as L

DEV = "cuda"
_IO = {"f32": torch.float32, "bf16": torch.bfloat16, "mxint8": L.MXINT8}
_IO_BYTES = {"f32": 4.0, "bf16": 2.0, "mxint8": 17.0 / 16.0}


def _case(kind, rows, K, N, rank, io="f32", w_bits=4, layers=1, heavy=False):
    """rows: tokens (calibration rows for ``calibrate``).  K, N: in- and out-features of ``linear`` and ``calibrate``; hidden
    and feed-forward size of ``layer`` and ``stack``.  heavy: Student-t weights and x50 outlier channels."""
    return {"kind": kind, "rows": rows, "K": K, "N": N, "rank": rank, "io": io, "w_bits": w_bits, "layers": layers, "heavy": heavy}


def listed():
    cases = {
        # one small layer at a small batch: nothing but launches and latency (the adapter-sized layer of the tests)
        "tiny_linear_m16": _case("linear", 16, 256, 256, 8),
        # one token of one sequence through a decoder layer, bf16 activations: interactive decoding
        "decode_layer_m1": _case("layer", 1, 4096, 11008, 32, io="bf16"),
        # one token through the linears of eight decoder layers as one batch: the decode leg of the benchmark's stack
        "decode_stack_m1": _case("stack", 1, 4096, 11008, 32, layers=8),
        # four tokens per step: a few sequences, or the drafts of speculative decoding
        "decode_layer_m4": _case("layer", 4, 4096, 11008, 32, io="bf16"),
        # sixteen sequences on the larger model with a larger rank, fp32 activations and heavy-tailed weights
        "decode_layer_m16": _case("layer", 16, 5120, 13824, 64, heavy=True),
        # a serving batch of 64 sequences
        "serve_layer_m64": _case("layer", 64, 5120, 13824, 32, io="bf16", heavy=True),
        # a ragged batch on a layer whose sizes fit no tile, quantised activations in and out
        "ragged_linear_m201": _case("linear", 201, 4112, 10992, 20, io="mxint8"),
        # a prefill chunk of 512 tokens with a rank of 128
        "chunk_layer_m512": _case("layer", 512, 5120, 13824, 128, heavy=True),
        # the prompt of 2048 tokens through a decoder layer, bf16 activations: ordinary prefill
        "prefill_layer_m2048": _case("layer", 2048, 4096, 11008, 32, io="bf16"),
        # the largest layer of the rank sweep: 4096 tokens, rank 256, fp32 activations
        "sweep_linear_m4096": _case("linear", 4096, 5120, 13824, 256, heavy=True),
        # 2-bit weights with their rank of 256, activations handed on quantised
        "w2_layer_m2048": _case("layer", 2048, 4096, 11008, 256, io="mxint8", w_bits=2),
        # preparing a layer for use: quantisation error, scaled truncated SVD, packing
        "calibrate_4096": _case("calibrate", 512, 4096, 4096, 32),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def draw(rng):
    """One more case of the same ranges."""
    def log_uniform(lo, hi):
        return lo * (hi / lo) ** rng.random()

    kind = rng.choices(("linear", "layer", "stack", "calibrate"), (8, 9, 2, 1))[0]
    rows = max(1, min(4096, int(round(log_uniform(0.7, 4096)))))
    rank = rng.choice((0, 8, 20, 32, 32, 48, 64, 100, 128, 256))
    io = rng.choice(("f32", "bf16", "bf16", "mxint8"))
    w_bits = rng.choice((4, 4, 4, 4, 2))
    heavy = rng.random() < 0.3
    if kind == "linear":
        K = 16 * int(log_uniform(16, 690))
        N = (16 if io == "mxint8" else 8) * int(log_uniform(32, 864))
        return _case(kind, rows, K, N, min(rank, K, N), io, w_bits, 1, heavy)
    if kind == "calibrate":
        return _case(kind, rng.choice((128, 512, 2048)), 256 * rng.randint(4, 16), 256 * rng.randint(4, 20),
                     rng.choice((8, 32, 32, 64)))
    hidden = 16 * int(log_uniform(64, 320))
    ffn = 16 * int(hidden * (2.5 + 0.5 * rng.random()) / 16)
    if kind == "stack":
        return _case(kind, rng.choice((1, 1, 2, 4, 8, 16)), hidden, ffn, rank, io, w_bits, rng.randint(2, 6), heavy)
    # no more work than the largest prefill layer
    rows = max(1, min(rows, int(2048 * (4 * 4096 ** 2 + 3 * 4096 * 11008) / (4 * hidden ** 2 + 3 * hidden * ffn))))
    return _case(kind, rows, hidden, ffn, rank, io, w_bits, 1, heavy)


def _shapes(case):
    """(K, N) of the case's linears in order, and the groups that go out as one call (index lists; a group of a ``layer`` shares
    one activation)."""
    K, N = case["K"], case["N"]
    if case["kind"] in ("linear", "calibrate"):
        return [(K, N)], [[0]]
    seven = [(K, K), (K, K), (K, K), (K, K), (K, N), (K, N), (N, K)]
    if case["kind"] == "layer":
        return seven, [[0, 1, 2], [3], [4, 5], [6]]
    return seven * case["layers"], [list(range(7 * case["layers"]))]


def _draw_weight(g, K, N, heavy):
    w = torch.randn((K, N), generator=g, device=DEV)
    if heavy:                                     # Student-t with 4 degrees of freedom, scaled to the same deviation
        chi = torch.zeros((K, N), device=DEV)
        for _ in range(4):
            chi.addcmul_(*(2 * [torch.randn((K, N), generator=g, device=DEV)]))
        w.div_(chi.div_(4.0).sqrt_()).mul_(0.5 ** 0.5)
    return w.mul_(0.02)


def _draw_activation(g, M, K, heavy):
    """N(0, 1) with a few outlier channels, as trained layers have them."""
    x = torch.randn((M, K), generator=g, device=DEV)
    n = max(1, int(K * (0.005 if heavy else 0.01)))
    x[:, torch.randperm(K, generator=g, device=DEV)[:n]] *= 50.0 if heavy else 20.0
    return x


def _draw_inputs(case, seed):
    """The numbers of a case: per linear (W, A, B) with A, B None at rank 0, and per linear its fp32 activation (one tensor where
    a group shares it)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    M, rank, heavy = case["rows"], case["rank"], case["heavy"]
    shapes, groups = _shapes(case)
    weights, Xs = [], [None] * len(shapes)
    for K, N in shapes:
        W = _draw_weight(g, K, N, heavy)
        A = B = None
        if rank and case["kind"] != "calibrate":  # factors of the magnitude that real ones have
            A = torch.randn((K, rank), generator=g, device=DEV) / K ** 0.5
            B = torch.randn((rank, N), generator=g, device=DEV) * (0.004 * (K ** 0.5 + N ** 0.5) / N ** 0.5)
        weights.append((W, A, B))
    for group in groups:
        shared = None
        for j in group:
            if shared is None or case["kind"] == "stack":
                shared = _draw_activation(g, M, shapes[j][0], heavy)
            Xs[j] = shared
    return g, weights, Xs


def prepare(case, seed):
    cfg = L.default_config()
    cfg.w_bits = case["w_bits"]
    M, rank, io = case["rows"], case["rank"], _IO[case["io"]]
    shapes, groups = _shapes(case)
    g, weights, drawn = _draw_inputs(case, seed)
    if case["kind"] == "calibrate":
        K, N = shapes[0]
        omega = torch.randn((N, L.factor_sketch_columns(K, N, rank)), generator=g, device=DEV)
        return {"kind": "calibrate", "W": weights[0][0], "samples": [drawn[0]], "rank": rank, "omega": omega, "cfg": cfg}

    packed, Xs, Ys, made = [], [], [], {}
    for (K, N), x in zip(shapes, drawn):
        packed.append(L.prepare_weights(*weights.pop(0), cfg))
        Ys.append(torch.zeros(L.mxint8_bytes(M, N), dtype=torch.uint8, device=DEV) if io == L.MXINT8
                  else torch.zeros((M, N), dtype=io, device=DEV))
        if id(x) not in made:
            made[id(x)] = L.to_mxint8(*L.quantize_activations(x, cfg)) if io == L.MXINT8 else x.to(io)
        Xs.append(made[id(x)])

    plan, need = [], max(L.workspace_bytes(M, K, N, rank, cfg) for K, N in shapes)
    for group in groups:
        if len(group) == 1:
            plan.append((group[0], None))
        else:
            calls = L.make_calls([(Xs[j], packed[j], Ys[j]) for j in group], io, io)
            need = max(need, L.batched_workspace_bytes(calls))
            plan.append((None, calls))
    ws = torch.zeros(need, dtype=torch.uint8, device=DEV)
    return {"kind": case["kind"], "io": io, "M": M, "packed": packed, "X": Xs, "Y": Ys, "plan": plan, "ws": ws}


def run(state):
    if state["kind"] == "calibrate":
        packed, A, B, _ = L.prepare_from_calibration(state["W"], state["samples"], state["rank"], state["omega"], state["cfg"])
        return {"packed": packed.buf, "A": A, "B": B}
    io, ws = state["io"], state["ws"]
    for j, calls in state["plan"]:
        if calls is None:
            L.linear_ex(state["X"][j], state["packed"][j], ws, state["Y"][j], io, M=state["M"])
        else:
            L.linear_batched_ex(calls, ws, io, io)
    return state["Y"]


def work(case):
    """Every stored operand, distinct input and output once; the products of the layer."""
    M, rank, b = case["rows"], case["rank"], _IO_BYTES[case["io"]]
    k_pad = (rank + 15) // 16 * 16
    shapes, groups = _shapes(case)
    if case["kind"] == "calibrate":
        # W, the calibration rows and the test matrix in; the packed buffer and the factors out; the ten products of the
        # error (K x N) with a matrix of rank + 16 columns that four rounds of subspace iteration consist of
        K, N = shapes[0]
        cols = rank + 16
        return {"bytes": 4.0 * (K * N + M * K + N * cols + rank * (K + N)) + 0.5625 * K * N + 1.0625 * k_pad * (K + N),
                "flops": 10 * 2.0 * K * N * cols}
    nbytes = flops = 0.0
    for group in groups:
        for i, j in enumerate(group):
            K, N = shapes[j]
            nbytes += (case["w_bits"] / 8.0 + 0.0625) * K * N + 1.0625 * (rank * K + k_pad * N) + b * M * N
            if i == 0 or case["kind"] == "stack":
                nbytes += b * M * K
            flops += 2.0 * M * ((K + rank) * N + K * rank)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Measured against fp64 on the stored operands: every product is exact in fp32 and most fp32 sums are too, so a Y
    # differs by 4e-9 (2-norm) and 2e-7 (single values) at most.  Another order of the fp32 sums stays within a few
    # 1e-7 of the largest terms; a bf16 or MXINT8 result then rounds the other way now and then, by one unit.
    if case["kind"] == "calibrate":               # fp64 sums throughout; the factors are rounded to fp32 at the end
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    return {"f32": {"rel": 1e-6, "max": 2e-5}, "bf16": {"rel": 1e-4, "max": 8e-3}, "mxint8": {"differ": 2e-4}}[case["io"]]


def _blocks(v, bits, dim):
    """MXINT: blocks of 16 along dim share e = floor(log2(max |v|)) in [-56, 55]; the mantissas are round-to-even of
    v / 2^(e - bits + 2), at most 2^(bits-1) - 1 in magnitude.  -> (mantissas and values as v lies, exponents), in fp64."""
    b = v.double().movedim(dim, -1).unflatten(-1, (-1, 16))
    amax = b.abs().amax(-1, keepdim=True)
    e = torch.where(amax > 0, torch.frexp(amax)[1].double() - 1, -56.0).clamp_(-56, 55)
    step = torch.exp2(e - (bits - 2))
    m = torch.round(b / step).clamp_(1 - 2 ** (bits - 1), 2 ** (bits - 1) - 1)
    return m.flatten(-2).movedim(-1, dim), (m * step).flatten(-2).movedim(-1, dim), e.squeeze(-1)


def exact(case, seed):
    if case["kind"] == "calibrate":               # singular vectors of a nearly flat spectrum: no such values
        return None
    _, weights, drawn = _draw_inputs(case, seed)
    rank, out = case["rank"], []
    for x in drawn:
        W, A, B = weights.pop(0)
        x = _blocks(x.bfloat16() if case["io"] == "bf16" else x, 8, 1)[1]
        y = x @ _blocks(W, case["w_bits"], 0)[1]
        if rank:
            pad = -rank % 16
            t = torch.nn.functional.pad(x @ _blocks(A, 8, 0)[1], (0, pad))
            y += _blocks(t, 8, 1)[1] @ _blocks(torch.nn.functional.pad(B, (0, 0, 0, pad)), 8, 0)[1]
        if case["io"] == "mxint8":
            m, _, e = _blocks(y, 8, 1)
            y = torch.cat([m.to(torch.int8).view(torch.uint8).flatten(), (e + 127).to(torch.uint8).flatten()])
        out.append(y)
    return out
