"""The prologue of larger batches with ranks above 64 (Section 3.1: T = X_q A_k as one integer contraction over digit planes)
against the oracle: T_q has to be bit-exact, whatever the blocks' exponents."""
import numpy as np
import pytest
import torch

import lqer_inputs as gen
import paper_2402_02446_b200 as L
from paper_2402_02446_b200 import binding
from helpers import exp_bytes, worst_ratio
from oracle import lqer as olqer

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _spread(v, axis, bits, seed):
    """v with every 16-block along `axis` scaled by a power of two from [-bits, bits]."""
    g = np.random.default_rng(seed)
    n = list(v.shape)
    n[axis] //= 16
    return (v * np.exp2(g.integers(-bits, bits + 1, size=n)).repeat(16, axis=axis)).astype(np.float32)


# row tiles that end inside a tile, K with a part of a panel of 128 (and a single 16-block), ranks that end inside a block or
# are cut into two column tiles, K ranges of one and of several panels
@pytest.mark.parametrize("M,K,k", [(129, 80, 72), (129, 272, 65), (130, 1040, 100), (257, 2048, 128), (300, 1200, 200), (1030, 512, 256)])
@pytest.mark.parametrize("wide", ["plain", "rows", "columns", "both"])
def test_t_is_exact_inside_and_outside_the_windows(M, K, k, wide):
    N = 264
    spec = gen.LayerSpec("digits", M=M, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=50.0, seed=900 + K)
    W = gen.make_weight(spec)
    A, B = gen.make_random_factors(spec)
    X = gen.make_activations(spec)
    if wide in ("rows", "both"):                       # every third row: block exponents over 25 binades
        X[::3] = _spread(X[::3], 1, 12, 1)
        X[1, :16] = 0.0
        X[2] = 0.0
        X[4, 3] = np.inf
    if wide in ("columns", "both"):
        A[:, ::5] = _spread(A[:, ::5], 0, 10, 2)
        A[:, 1] = 0.0
    P, Pg = olqer.prepare_weights(W, A, B), L.prepare_weights(_t(W), _t(A), _t(B))
    ref = olqer.forward(X, P)
    ws = L.new_workspace(M, Pg)
    L.set_path(binding.PATH_TENSOR_PROLOGUE)           # whatever the amount of work
    try:
        Tm, Te = L.project_lowrank(_t(X), Pg, ws)
        Y = L.linear(_t(X), Pg, ws).cpu().numpy()
    finally:
        L.set_path(binding.PATH_AUTO)
    assert L.poll_status(ws) == 0
    assert np.array_equal(Tm.cpu().numpy(), ref.Tm)
    assert np.array_equal(Te.cpu().numpy(), exp_bytes(ref.Te))
    assert np.all(Y[ref.tol == 0.0] == 0.0)            # a row of zeros
    ref.tol[ref.tol == 0.0] = 1.0
    assert worst_ratio(Y, ref) <= 1.0
    # the other prologue of these ranks gives the same result
    L.set_path(binding.PATH_TENSOR)
    try:
        assert np.array_equal(L.linear(_t(X), Pg, ws).cpu().numpy(), Y)
    finally:
        L.set_path(binding.PATH_AUTO)
    Pg.release()


# a row's blocks lie in windows of nine exponents below its largest or above its smallest (three of them, two above 32768 K)
# or below those: block exponents at both edges of every window, in every block, in two blocks of a panel, in the last only
@pytest.mark.parametrize("M,K,k,a_bits", [(140, 1040, 80, 8), (257, 4112, 136, 6), (129, 32784, 72, 8), (1030, 512, 256, 8)])
def test_windows_beyond_the_first(M, K, k, a_bits):
    N, g = 264, np.random.default_rng(K)
    spec = gen.LayerSpec("windows", M=M, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.0, outlier_scale=1.0, seed=930 + k)
    W = gen.make_weight(spec)
    A, B = gen.make_random_factors(spec)
    A[:16 * (K // 32)] *= 2.0 ** -10                         # columns with blocks outside theirs
    X = g.uniform(1.0, 2.0, (M, K)).astype(np.float32) * g.choice((-1.0, 1.0), (M, K)).astype(np.float32)
    e = np.zeros((M, K // 16))
    for r in range(M):
        low = (8, 9, 17, 18, 26, 27, 35, 50)[r % 8]
        kind = r // 8 % 4
        if kind == 0: e[r] = -g.integers(0, low + 1, K // 16)
        elif kind == 1: e[r, 9:11] = -low if r % 3 else low
        elif kind == 2: e[r, -1] = low if r % 3 else -low
        else: e[r] = -g.choice((0, 8, 9, 17, 18, 26, 27, 44), K // 16)
    X *= np.exp2(e).repeat(16, axis=1).astype(np.float32)
    cfg = L.default_config()
    cfg.a_bits = a_bits
    P, Pg = olqer.prepare_weights(W, A, B), L.prepare_weights(_t(W), _t(A), _t(B), cfg)
    ref = olqer.forward(X, P, a_bits=a_bits)
    ws = L.new_workspace(M, Pg)
    L.set_path(binding.PATH_TENSOR_PROLOGUE)
    try:
        Tm, Te = L.project_lowrank(_t(X), Pg, ws)
        Y = L.linear(_t(X), Pg, ws).cpu().numpy()
    finally:
        L.set_path(binding.PATH_AUTO)
    assert L.poll_status(ws) == 0
    assert np.array_equal(Te.cpu().numpy(), exp_bytes(ref.Te))
    assert np.array_equal(Tm.cpu().numpy(), ref.Tm)
    assert worst_ratio(Y, ref) <= 1.0
    Pg.release()


@pytest.mark.parametrize("x_type", ["f32", "bf16", "mxint8"])
def test_layers_that_share_an_activation_equal_single_calls(x_type):
    # three calls on one X, one on another, ranks of two widths: one group; each result is the single call's, bit for bit
    M = 300
    specs = [gen.LayerSpec(f"share{i}", M=M, K=2064, N=n, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=950 + i)
             for i, (n, k) in enumerate([(256, 80), (520, 256), (264, 112), (256, 80)])]
    packs = []
    for s in specs:
        A, B = gen.make_random_factors(s)
        packs.append(L.prepare_weights(_t(gen.make_weight(s)), _t(A), _t(B)))
    Xs = [_t(gen.make_activations(specs[0])), _t(gen.make_activations(specs[3]))]
    dt = {"f32": torch.float32, "bf16": torch.bfloat16, "mxint8": L.MXINT8}[x_type]
    Xs = [L.to_mxint8(*L.quantize_activations(x)) if dt == L.MXINT8 else x.to(dt) for x in Xs]
    Xc = [Xs[0], Xs[0], Xs[1], Xs[0]]
    Ys = [torch.full((M, s.N), float("nan"), device=DEV) for s in specs]
    calls = L.make_calls(list(zip(Xc, packs, Ys)), dt, torch.float32)
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    for _ in range(2):
        L.linear_batched_ex(calls, ws, dt, torch.float32)
    assert L.poll_status(ws) == 0
    for x, Pg, y in zip(Xc, packs, Ys):
        assert torch.equal(L.linear_ex(x, Pg, ws, M=M), y)
        Pg.release()


def test_low_ranks_on_one_activation():
    # ranks up to 64 take the digit planes where large layers share an activation; single calls the fp64-scaled prologue
    M, K = 1100, 4112
    specs = [gen.LayerSpec(f"low{i}", M=M, K=K, N=264, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=50.0, seed=980 + i)
             for i, k in enumerate((32, 40, 64))]
    layers = []
    for s in specs:
        W, (A, B) = gen.make_weight(s), gen.make_random_factors(s)
        layers.append((olqer.prepare_weights(W, A, B), L.prepare_weights(_t(W), _t(A), _t(B))))
    X = gen.make_activations(specs[0])
    X[5::7] = _spread(X[5::7], 1, 9, 3)
    x = _t(X)
    Ys = [torch.full((M, s.N), float("nan"), device=DEV) for s in specs]
    calls = L.make_calls([(x, Pg, y) for (_, Pg), y in zip(layers, Ys)])
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    L.linear_batched(calls, ws)
    assert L.poll_status(ws) == 0
    rows = np.arange(0, M, 53)
    for (P, Pg), y in zip(layers, Ys):
        assert torch.equal(L.linear(x, Pg, ws), y)
        assert worst_ratio(y.cpu().numpy()[rows], olqer.forward(X[rows], P)) <= 1.0
        Pg.release()


def test_a_workspace_without_room_for_the_planes_is_taken_as_before():
    spec = gen.LayerSpec("tight", M=300, K=4112, N=264, k=128, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=970)
    A, B = gen.make_random_factors(spec)
    Pg = L.prepare_weights(_t(gen.make_weight(spec)), _t(A), _t(B))
    X = _t(gen.make_activations(spec))
    Y = L.linear(X, Pg, L.new_workspace(spec.M, Pg))
    least = 168192 + (spec.M * (4160 + 128) * 2 + 255) // 256 * 256       # the head and [X_q | T_q]
    ws = torch.zeros(least, dtype=torch.uint8, device=DEV)
    assert torch.equal(L.linear(X, Pg, ws), Y) and L.poll_status(ws) == 0
    with pytest.raises(binding.LqerError):
        L.linear(X, Pg, ws[: least - 256])
    Pg.release()


# ranks whose own prologue needs less scratch than the planes: 48 (none at all), 32 at many row tiles, 16 at a long K; and
# layers on activations of their own, whose planes need more than two slices have
@pytest.mark.parametrize("M,K,k,shared", [(2048, 4096, 48, True), (8192, 4096, 32, True), (4096, 5120, 16, True), (1030, 2048, 128, False)])
def test_the_advised_workspace_has_room_for_the_planes(M, K, k, shared):
    N = 256
    specs = [gen.LayerSpec(f"room{i}", M=M, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=990 + i) for i in range(2)]
    packs = [L.prepare_weights(_t(gen.make_weight(s)), *map(_t, gen.make_random_factors(s))) for s in specs]
    Xs = [torch.randn((M, K), generator=torch.Generator(device=DEV).manual_seed(k + i), device=DEV) for i in range(2)]
    Xs[1] = Xs[0] if shared else Xs[1]
    Ys = [torch.full((M, N), float("nan"), device=DEV) for _ in specs]
    calls = L.make_calls(list(zip(Xs, packs, Ys)))
    single = [L.linear(x, P, L.new_workspace(M, P)) for x, P in zip(Xs, packs)]

    def launches(nbytes):
        ws = torch.zeros(nbytes, dtype=torch.uint8, device=DEV)
        before = L.launch_count()
        L.linear_batched(calls, ws)
        n = L.launch_count() - before
        assert L.poll_status(ws) == 0
        assert all(torch.equal(y, s) for y, s in zip(Ys, single))
        return n
    assert launches(L.batched_workspace_bytes(calls)) == 4       # three for the planes, one GEMM
    if not shared:                                               # two bare Xcats: taken, as before there were planes
        assert launches(168192 + 2 * M * (K + k) * 2) == 3
    for P in packs:
        P.release()
