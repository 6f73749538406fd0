"""The sum of a tile's K chunks in the small-batch GEMM (Section 3.1: Y = X_q W_q + T_q B_q), which the CTAs of its chunks share:
few and many rows, up to 21 chunks, a missing 128-column half, and a launch whose CTAs have several chunks each."""
import numpy as np
import pytest
import torch

import lqer_inputs as gen
import paper_2402_02446_b200 as L
from oracle import lqer as olqer
from helpers import worst_ratio

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _layer(K, N, k, M, seed):
    spec = gen.LayerSpec("sums", M=M, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=seed)
    W = gen.make_weight(spec)
    A, B = gen.make_random_factors(spec)
    return spec, olqer.prepare_weights(W, A, B), L.prepare_weights(_t(W), _t(A), _t(B))


# 21 chunks of two tiles: four shares of the rows with 17 tokens, more shares than rows need with 128; 2 chunks: one share, two
@pytest.mark.parametrize("K,N", [(11008, 264), (1088, 400)])
@pytest.mark.parametrize("M", [17, 47, 49, 128])
def test_shares_of_the_rows(M, K, N):
    spec, P, Pg = _layer(K, N, 40, M, 1500 + M)
    X = gen.make_activations(spec)
    ref = olqer.forward(X, P)
    ws = L.new_workspace(M, Pg)
    ws[168192:] = 0xFF                                  # scratch holds NaN patterns: nothing unwritten may be read
    first = None
    for _ in range(3):                                  # (the second call finds the counters as the first left them)
        Y = L.linear(_t(X), Pg, ws)
        assert L.poll_status(ws) == 0
        assert worst_ratio(Y.cpu().numpy(), ref) <= 1.0
        first = Y.clone() if first is None else first
        assert torch.equal(Y, first)
    Pg.release()


@pytest.mark.parametrize("M", [20, 100])
def test_ctas_with_several_chunks(M):
    # 150 tiles of 129 slabs: cut into two chunks each, three rounds of the SMs, so that most chunks are not their CTA's last
    spec, P, Pg = _layer(8192, 2424, 40, M, 1600 + M)
    X = gen.make_activations(spec)
    ref = olqer.forward(X, P)
    x = _t(X)
    Ys = [torch.full((M, spec.N), float("nan"), device=DEV) for _ in range(15)]
    calls = L.make_calls([(x, Pg, y) for y in Ys])
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    for _ in range(2):
        before = L.launch_count()
        L.linear_batched(calls, ws)
        assert L.poll_status(ws) == 0 and L.launch_count() - before == 2
    assert worst_ratio(Ys[0].cpu().numpy(), ref) <= 1.0
    for y in Ys[1:]:
        assert torch.equal(y, Ys[0])
    Pg.release()
