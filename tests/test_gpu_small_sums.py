"""The sum of a tile's K chunks in the small-batch GEMM (Section 3.1: Y = X_q W_q + T_q B_q), which the CTAs of its chunks share:
few and many rows, up to 21 chunks, a missing 128-column half, a launch whose CTAs have several chunks each, and one whose CTAs have all
chunks of a tile each; and how far layers that share a launch may be from 64 bits."""
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


def _groups(K, N, k, n, g, one_sign=False):
    draw = lambda *s: torch.randn(s, generator=g, device=DEV)
    W, A, B = [], [], []
    for _ in range(n):
        w = draw(K, N) * 0.02
        W.append(w.abs() if one_sign else w)
        A.append(draw(K, k) / K ** 0.5)
        B.append(draw(k, N) * 0.01)
    return W, A, B, [L.prepare_weights(*f) for f in zip(W, A, B)]


def _oracle(W, A, B, cols):
    h = lambda a: a.cpu().numpy()
    return olqer.prepare_weights(h(W[:, cols]), h(A), h(B[:, cols]))         # (columns are independent)


# Two layers of 76 tiles (the last with one half) and three chunks: 228 items where 76 CTAs can take a tile each.  Two of 52 tiles and five chunks: two
# CTAs take three and two chunks of each.  Three of 51 tiles: five chunks would do, two CTAs take three of six each.
@pytest.mark.parametrize("M,K,N,n", [(17, 2048, 9592, 2), (32, 4096, 9592, 2), (33, 4096, 9592, 2), (64, 4096, 9592, 2), (65, 4096, 9592, 2), (128, 4096, 9592, 2),
                                     (17, 4096, 6408, 2), (64, 4096, 6408, 2), (128, 4096, 6408, 2), (20, 4352, 4232, 3), (128, 4352, 4232, 3)])
def test_ctas_with_runs_of_a_tiles_chunks(M, K, N, n):
    k = 40
    g = torch.Generator(device=DEV)
    g.manual_seed(1700 + M)
    W, A, B, P = _groups(K, N, k, n, g)
    X = torch.randn((M, K), generator=g, device=DEV)
    cols = torch.cat([torch.arange(0, 64), torch.arange(N - 136, N)]).to(DEV)
    lone = [L.linear(X, p, L.new_workspace(M, p)) for p in P]
    oracle = [_oracle(w, a, b, cols) for w, a, b in zip(W, A, B)]
    for dtype in (torch.float32, torch.bfloat16):
        Ys = [torch.full((M, N), float("nan"), device=DEV, dtype=dtype) for _ in P]
        calls = L.make_calls([(X, p, y) for p, y in zip(P, Ys)], torch.float32, dtype)
        ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
        ws[168192:] = 0xFF                              # scratch holds NaN patterns: nothing unwritten may be read
        for _ in range(2):
            before = L.launch_count()
            L.linear_batched_ex(calls, ws, torch.float32, dtype)
            assert L.poll_status(ws) == 0 and L.launch_count() - before == 2
            if dtype == torch.float32:
                for y, o in zip(Ys, oracle):
                    assert worst_ratio(y[:, cols].cpu().numpy(), olqer.forward(X.cpu().numpy(), o)) <= 1.0
                whole = [y.clone() for y in Ys]
                if n == 2:                              # the layer alone has the same cut, one CTA to a chunk
                    assert all(torch.equal(y, z) for y, z in zip(Ys, lone))
            assert all(torch.equal(y, z.to(dtype)) for y, z in zip(Ys, whole))
    for p in P:
        p.release()


@pytest.mark.parametrize("K,N,n", [(4096, 11008, 2), (1024, 1024, 3), (1024, 2816, 2)])
@pytest.mark.parametrize("M", [17, 64, 128])
def test_shared_launches_are_no_further_off_than_the_layer_alone(M, K, N, n):
    # one sign and block exponents over a dozen binades: no fp32 sum is exact, and the accumulators of tensor memory cut off what does not
    # fit, so a longer chain is further off (4096 x 11008 in one piece 7 times).  Half as much again is left for the draw of the inputs.
    g = torch.Generator(device=DEV)
    g.manual_seed(1800 + M)
    W, A, B, P = _groups(K, N, 32, n, g, one_sign=True)
    X = torch.randn((M, K), generator=g, device=DEV).abs()
    X = X * torch.exp2(torch.randint(-6, 7, (M, K // 16), generator=g, device=DEV).float()).repeat_interleave(16, 1)
    cols = torch.arange(0, N, max(N // 192, 1)).to(DEV)
    ref = olqer.forward(X.cpu().numpy(), _oracle(W[0], A[0], B[0], cols)).Y
    error = lambda y: float(np.linalg.norm(y[:, cols].double().cpu().numpy() - ref) / np.linalg.norm(ref))
    ws = L.new_workspace(M, P[0])
    alone = error(L.linear(X, P[0], ws))
    Ys = [torch.empty((M, N), device=DEV) for _ in P]
    calls = L.make_calls([(X, p, y) for p, y in zip(P, Ys)])
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    L.linear_batched(calls, ws)
    assert L.poll_status(ws) == 0
    assert 0.0 < error(Ys[0]) <= 1.5 * alone, (error(Ys[0]), alone)
    for p in P:
        p.release()
