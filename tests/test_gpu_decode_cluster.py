"""Batches of 3 to 16 rows in one launch: a cluster of CTAs per range of columns, the contraction shared by its CTAs.

Sizes sit at the edges of what the kernel cuts: contractions that give a CTA one slab, half a step or a ragged last block, fewer columns than
a tile of 128, one and several tiles to a cluster with a nearly empty last one, ranks of no, one, several and sixteen blocks, and both
sides of the eight-token tile.
"""
import numpy as np
import pytest
import torch

import lqer_inputs as gen
import paper_2402_02446_b200 as L
from paper_2402_02446_b200 import binding
from oracle import lqer as olqer
from helpers import worst_ratio

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _layer(K, N, k, seed, w_bits=4):
    spec = gen.LayerSpec("cluster", M=16, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=seed)
    W = gen.make_weight(spec)
    A, B = gen.make_random_factors(spec) if k else (None, None)
    cfg = L.default_config()
    cfg.w_bits = w_bits
    return spec, olqer.prepare_weights(W, A, B, w_bits=w_bits), L.prepare_weights(_t(W), *((_t(A), _t(B)) if k else (None, None)), cfg)


SHAPES = [
    # K, N, k, w_bits
    (16, 8, 0, 4), (64, 24, 5, 4), (208, 264, 16, 4), (1024, 8704, 16, 4), (1040, 20008, 24, 4), (2112, 264, 72, 4),
    (1152, 1032, 256, 4), (4112, 520, 40, 4), (1040, 648, 136, 2), (304, 4104, 20, 2),
]


@pytest.mark.parametrize("K,N,k,w_bits", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_rows_3_to_16_against_the_oracle(K, N, k, w_bits):
    spec, P, Pg = _layer(K, N, k, 901, w_bits)
    X = gen.make_activations(spec, M=16)
    for M in (3, 8, 9, 16):
        ref = olqer.forward(X[:M], P, w_bits=w_bits)
        Xg, ws = _t(X[:M]), L.new_workspace(M, Pg)
        before = L.launch_count()
        Y = L.linear(Xg, Pg, ws)
        assert L.launch_count() - before == 1
        again = L.linear(Xg, Pg, ws)                       # the counters are zero again
        assert L.poll_status(ws) == 0
        assert torch.equal(Y, again)
        assert worst_ratio(Y.cpu().numpy(), ref) <= 1.0, M
    Pg.release()


@pytest.mark.parametrize("K,k", [(1040, 16), (13824, 64), (4096, 256)])
@pytest.mark.parametrize("M", [3, 4, 8, 16])
def test_rounded_sums_are_no_further_off_than_the_other_kernels(M, K, k):
    # one sign and block exponents over a dozen binades: no fp32 sum is exact.  Against the column-owner kernel (up to four rows: dot
    # products added by rounded fp32 operations) or the tensor-memory GEMM, both on path 2; half as much again is left for the
    # draw of the inputs (the kernels' own ratios are 0.5 to 1.0).
    spec = gen.LayerSpec("rounds", M=M, K=K, N=520, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=904)
    W = np.abs(gen.make_weight(spec))
    A, B = gen.make_random_factors(spec)
    P, Pg = olqer.prepare_weights(W, A, B), L.prepare_weights(_t(W), _t(A), _t(B))
    X = np.abs(gen.make_activations(spec)) * np.exp2(np.random.default_rng(9).integers(-6, 7, size=(M, K // 16))).repeat(16, axis=1).astype(np.float32)
    ref = olqer.forward(X, P)
    ws = L.new_workspace(M, Pg)
    error = {}
    for path in (binding.PATH_AUTO, binding.PATH_DECODE):
        L.set_path(path)
        try:
            y = L.linear(_t(X), Pg, ws).cpu().numpy().astype(np.float64)
        finally:
            L.set_path(binding.PATH_AUTO)
        assert L.poll_status(ws) == 0
        error[path] = np.linalg.norm(y - ref.Y) / np.linalg.norm(ref.Y)
    assert 0.0 < error[binding.PATH_AUTO] <= 1.5 * error[binding.PATH_DECODE], error
    Pg.release()


@pytest.mark.parametrize("M", [3, 16])
def test_types_at_the_boundary(M):
    # bf16 X is the fp32 value it denotes; MXINT8 in and out agree with quantising outside
    spec, P, Pg = _layer(1040, 1040, 40, 902)
    X = _t(gen.make_activations(spec, M=M))
    ws = L.new_workspace(M, Pg)
    Xb = X.bfloat16()
    y = L.linear_ex(Xb.float(), Pg, ws)
    assert torch.equal(L.linear_ex(Xb, Pg, ws), y)
    assert torch.equal(L.linear_ex(Xb, Pg, ws, out_dtype=torch.bfloat16), y.bfloat16())
    cfg = L.default_config()
    mx = L.to_mxint8(*L.quantize_activations(X, cfg))
    y = L.linear(X, Pg, ws)
    assert torch.equal(L.linear_ex(mx, Pg, ws, M=M), y)
    got = L.linear_ex(mx, Pg, ws, out_dtype=L.MXINT8, M=M)
    assert torch.equal(got, L.to_mxint8(*L.quantize_activations(y, cfg)))
    assert L.poll_status(ws) == 0
    Pg.release()


@pytest.mark.parametrize("M", [4, 12])
def test_groups_share_one_launch(M):
    # two to four neighbours, of one shape and of several; also as replays of a captured graph on new activations
    shapes = [(1040, 520, 40), (512, 1032, 0), (2112, 264, 72), (1040, 648, 256)]
    layers = [_layer(*s, 903 + i) for i, s in enumerate(shapes)]
    for pick in ((0, 0), (0, 3, 0), (0, 1, 2, 3)):
        Xs = [_t(gen.make_activations(layers[j][0], M=M)) + 0.125 * i for i, j in enumerate(pick)]
        Ys = [torch.full((M, layers[j][0].N), float("nan"), device=DEV) for j in pick]
        calls = L.make_calls([(x, layers[j][2], y) for x, j, y in zip(Xs, pick, Ys)])
        ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
        before = L.launch_count()
        L.linear_batched(calls, ws)
        assert L.launch_count() - before == 1
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            L.linear_batched(calls, ws, stream=torch.cuda.current_stream())
        for rep in range(3):
            for x in Xs:
                x.mul_(-1.5)
            graph.replay()
            torch.cuda.synchronize()
            assert L.poll_status(ws) == 0
            for x, j, y in zip(Xs, pick, Ys):
                assert worst_ratio(y.cpu().numpy(), olqer.forward(x.cpu().numpy(), layers[j][1])) <= 1.0, (pick, rep)
    for l in layers:
        l[2].release()


def test_streams_with_a_workspace_each():
    # four streams of calls whose T comes from several clusters (one block of ranks each, two, four), beside a stream that keeps the SMs
    # busy: nobody waits for good, and every result is the lone call's
    shapes = [(4096, 1032, 256), (4096, 1032, 64), (12288, 520, 256), (1040, 4104, 256)]
    layers = [_layer(*s, 905 + i) for i, s in enumerate(shapes)]
    rows = (3, 16, 8, 5)
    Xs = [_t(gen.make_activations(l[0], M=m)) for l, m in zip(layers, rows)]
    want = [L.linear(x, l[2], L.new_workspace(m, l[2])) for x, l, m in zip(Xs, layers, rows)]
    for w, x, l in zip(want, Xs, layers):
        assert worst_ratio(w.cpu().numpy(), olqer.forward(x.cpu().numpy(), l[1])) <= 1.0
    streams = [torch.cuda.Stream(priority=-(i % 2)) for i in range(4)]
    spaces = [[L.new_workspace(m, l[2]) for m, l in zip(rows, layers)] for _ in streams]
    Ys = [[[torch.full_like(w, float("nan")) for w in want] for _ in range(12)] for _ in streams]
    busy, a = torch.cuda.Stream(), torch.zeros((8192, 8192), device=DEV)
    torch.cuda.synchronize()
    for rep in range(12):
        with torch.cuda.stream(busy):
            torch.add(a, 1.0, out=a)
        for i, s in enumerate(streams):
            for j in range(4):
                q = (i + j) % 4
                L.linear(Xs[q], layers[q][2], spaces[i][q], Ys[i][rep][q], stream=s)
    torch.cuda.synchronize()
    for i in range(4):
        assert all(L.poll_status(w) == 0 for w in spaces[i])
        for got in Ys[i]:
            assert all(torch.equal(y, w) for y, w in zip(got, want))
    for l in layers:
        l[2].release()


def test_replays_of_a_launch_whose_t_comes_from_several_clusters():
    # long K and a high rank: four clusters form T, which reaches the others through global memory and counters; captured
    spec, P, Pg = _layer(12288, 520, 256, 909)
    x, y, ws = torch.zeros((8, spec.K), device=DEV), torch.zeros((8, spec.N), device=DEV), L.new_workspace(8, Pg)
    L.linear(x, Pg, ws, y)
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=stream):
        L.linear(x, Pg, ws, y, stream=torch.cuda.current_stream())
    for rep in range(3):
        X = gen.make_activations(spec, M=8) * np.float32(1 + rep)
        x.copy_(_t(X))
        graph.replay()
        torch.cuda.synchronize()
        assert L.poll_status(ws) == 0
        assert worst_ratio(y.cpu().numpy(), olqer.forward(X, P)) <= 1.0, rep
    Pg.release()


def test_many_streams_of_launches_whose_t_comes_from_several_clusters():
    # ten streams of two priorities, ranks of 256: their clusters that form T are more than the device has places.  Nobody waits for good.
    spec, P, Pg = _layer(12288, 520, 256, 910)
    X = _t(gen.make_activations(spec, M=8))
    want = L.linear(X, Pg, L.new_workspace(8, Pg))
    assert worst_ratio(want.cpu().numpy(), olqer.forward(X.cpu().numpy(), P)) <= 1.0
    streams = [torch.cuda.Stream(priority=-(i % 2)) for i in range(10)]
    spaces = [L.new_workspace(8, Pg) for _ in streams]
    Ys = [[torch.full_like(want, float("nan")) for _ in range(20)] for _ in streams]
    torch.cuda.synchronize()
    for rep in range(20):
        for s, w, ys in zip(streams, spaces, Ys):
            L.linear(X, Pg, w, ys[rep], stream=s)
    torch.cuda.synchronize()
    assert all(L.poll_status(w) == 0 for w in spaces)
    assert all(torch.equal(y, want) for ys in Ys for y in ys)
    Pg.release()
