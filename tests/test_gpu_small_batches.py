"""The small-batch GEMM with the weights in tensor memory and its prologue (Section 3.1: Y = X_q W_q + T_q B_q) against the
oracle, at the edges of its tiles: token counts around the MMA widths, batches of slabs and steps that end early, a missing
128-column half, rank slabs that end inside a block of 64, both weight widths, every output type."""
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


def _layer(spec, w_bits):
    cfg = L.default_config()
    cfg.w_bits = w_bits
    W = gen.make_weight(spec)
    A, B = gen.make_random_factors(spec) if spec.k else (None, None)
    g = (lambda v: None if v is None else _t(v))
    return olqer.prepare_weights(W, A, B, w_bits=w_bits), L.prepare_weights(_t(W), g(A), g(B), cfg)


# slabs of 64 K: 1; 2 + a part; 5 (a batch of four, then one); 17 (cut into chunks); ranks: none, one block, a slab and a
# part, two slabs, four
@pytest.mark.parametrize("K,N,k", [(64, 16, 0), (144, 136, 16), (320, 264, 72), (1088, 400, 128), (528, 1032, 200)])
@pytest.mark.parametrize("M", [5, 16, 17, 32, 33, 49, 64, 65, 113, 128])
def test_token_counts_and_tile_edges(M, K, N, k):
    w_bits = 2 if (M + K) % 3 == 0 else 4
    spec = gen.LayerSpec("tiles", M=M, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.02, outlier_scale=20.0, seed=1100 + K + M)
    P, Pg = _layer(spec, w_bits)
    X = gen.make_activations(spec)
    ref = olqer.forward(X, P, w_bits=w_bits)
    ws = L.new_workspace(M, Pg)
    ws[168192:] = 0xFF                                  # scratch holds NaN patterns: nothing unwritten may be read
    # up to 16 rows a lone call takes the cluster kernel by itself (test_gpu_decode_cluster.py)
    L.set_path(binding.PATH_SMALL_TMEM if M <= 16 else binding.PATH_AUTO)
    try:
        for _ in range(2):
            Y = L.linear(_t(X), Pg, ws)
            assert L.poll_status(ws) == 0
            assert worst_ratio(Y.cpu().numpy(), ref) <= 1.0
        assert torch.equal(L.linear_ex(_t(X), Pg, ws, out_dtype=torch.bfloat16), Y.to(torch.bfloat16))
        if k:
            Tm, Te = L.project_lowrank(_t(X), Pg, ws)
            assert np.array_equal(Tm.cpu().numpy(), ref.Tm) and np.array_equal(Te.cpu().numpy(), exp_bytes(ref.Te))
        if N % 16 == 0:
            m8, e8 = L.split_mxint8(L.linear_ex(_t(X), Pg, ws, out_dtype=L.MXINT8), M, N)
            qm, qe = L.quantize_activations(Y)          # the codes of the same path's fp32 result
            assert torch.equal(m8, qm) and torch.equal(e8, qe)
    finally:
        L.set_path(binding.PATH_AUTO)
    Pg.release()


@pytest.mark.parametrize("M", [20, 64, 100])
def test_layers_of_one_launch(M):
    # five layers of three shapes in one launch: the cut of their tiles differs from single calls', the sums agree to rounding
    specs = [gen.LayerSpec(f"one{i}", M=M, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=1300 + i)
             for i, (K, N, k) in enumerate([(1024, 640, 40), (1024, 640, 40), (2112, 264, 16), (512, 1288, 100), (1024, 640, 0)])]
    layers = [_layer(s, 4) for s in specs]
    Xs = [_t(gen.make_activations(s)) for s in specs]
    Ys = [torch.full((M, s.N), float("nan"), device=DEV) for s in specs]
    calls = L.make_calls([(x, lay[1], y) for x, lay, y in zip(Xs, layers, Ys)])
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    for _ in range(2):
        L.linear_batched(calls, ws)
        assert L.poll_status(ws) == 0
    for s, (P, Pg), x, y in zip(specs, layers, Xs, Ys):
        assert worst_ratio(y.cpu().numpy(), olqer.forward(x.cpu().numpy(), P)) <= 1.0, s.name
        Pg.release()


def test_wide_exponents_alone_and_in_company():
    # block exponents over 50 binades: the fp64 sums of T round, and a launch of several layers groups them differently (the
    # cluster that shares a K range depends on all of its layers); both stay within the tolerance
    M = 20
    specs = [gen.LayerSpec(f"wide{i}", M=M, K=K, N=264, k=40, calib_rows=32, outlier_frac=0.0, outlier_scale=1.0, seed=1400 + i)
             for i, K in enumerate((4096, 1024, 4096, 2112))]
    layers = [_layer(s, 4) for s in specs]
    g = np.random.default_rng(5)
    Xs = [(gen.make_activations(s) * np.exp2(g.integers(-40, 11, (M, s.K // 16))).repeat(16, axis=1)).astype(np.float32) for s in specs]
    Ys = [torch.full((M, s.N), float("nan"), device=DEV) for s in specs]
    xs = [_t(x) for x in Xs]
    calls = L.make_calls([(x, lay[1], y) for x, lay, y in zip(xs, layers, Ys)])
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    L.linear_batched(calls, ws)
    assert L.poll_status(ws) == 0
    for (P, Pg), X, x, y in zip(layers, Xs, xs, Ys):
        ref = olqer.forward(X, P)
        assert worst_ratio(y.cpu().numpy(), ref) <= 1.0
        assert worst_ratio(L.linear(x, Pg, ws).cpu().numpy(), ref) <= 1.0
        Tm, Te = L.project_lowrank(x, Pg, ws)
        assert np.array_equal(Tm.cpu().numpy(), ref.Tm) and np.array_equal(Te.cpu().numpy(), exp_bytes(ref.Te))
        Pg.release()
