"""The cut of the cluster kernel (3 to 16 rows): tiles of 128 columns, stages of 128 K, one cluster's T or every cluster's own.

Sizes: a last tile of one column octet, an odd last slab, fewer stages than consumer warps take in turn, more tiles than clusters with
fewer of them for the clusters that form T, rings shorter and longer than a CTA's stages, and both sides of the rules that let a
cluster form all of T itself (128 ranks, ten stages, eight blocks a warp).
"""
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


@pytest.mark.parametrize("K,N,k,w_bits", [
    (128, 136, 128, 4), (192, 136, 129, 4), (208, 8, 8, 4), (256, 1288, 16, 2), (1040, 136, 40, 4), (4096, 1032, 16, 4),
    (4096, 9224, 32, 4), (2064, 20488, 72, 2), (11008, 392, 32, 4),
])
def test_cuts_against_the_oracle(K, N, k, w_bits):
    spec = gen.LayerSpec("cut", M=16, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=941)
    W = gen.make_weight(spec)
    A, B = gen.make_random_factors(spec)
    cfg = L.default_config()
    cfg.w_bits = w_bits
    P, Pg = olqer.prepare_weights(W, A, B, w_bits=w_bits), L.prepare_weights(_t(W), _t(A), _t(B), cfg)
    X = gen.make_activations(spec, M=16)
    for M in (3, 8, 9, 16):
        ref = olqer.forward(X[:M], P, w_bits=w_bits)
        Xg, ws = _t(X[:M]), L.new_workspace(M, Pg)
        before = L.launch_count()
        Y = L.linear(Xg, Pg, ws)
        assert L.launch_count() - before == 1
        again = L.linear(Xg, Pg, ws)
        assert L.poll_status(ws) == 0
        assert torch.equal(Y, again)
        assert worst_ratio(Y.cpu().numpy(), ref) <= 1.0, M
    Pg.release()


# rings of 5, 4, 17 and 20 slots for 40 to 72 stages: filled many times over, and no multiple of the three consumers that take them in turn
@pytest.mark.parametrize("M,K,N,k,w_bits", [(16, 11008, 11008, 32, 4), (16, 12288, 11008, 32, 4), (4, 4096, 20488, 32, 4), (8, 4096, 25096, 0, 2)])
def test_rings_that_are_filled_again(M, K, N, k, w_bits):
    g = torch.Generator(device=DEV)
    g.manual_seed(942)
    draw = lambda *s: torch.randn(s, generator=g, device=DEV)
    W, A, B, X = draw(K, N) * 0.02, draw(K, k) / K ** 0.5, draw(k, N) * 0.01, draw(M, K)
    cfg = L.default_config()
    cfg.w_bits = w_bits
    Pg = L.prepare_weights(W, A if k else None, B if k else None, cfg)
    cols = torch.cat([torch.arange(0, 72), torch.arange(N // 2 - 64, N // 2 + 64), torch.arange(N - 136, N)]).to(DEV)
    h = lambda a: a.cpu().numpy()
    P = olqer.prepare_weights(h(W[:, cols]), h(A) if k else None, h(B[:, cols]) if k else None, w_bits=w_bits)    # columns are independent
    del W
    ws = L.new_workspace(M, Pg)
    before = L.launch_count()
    Y = L.linear(X, Pg, ws)
    assert L.launch_count() - before == 1
    assert L.poll_status(ws) == 0
    assert worst_ratio(h(Y[:, cols]), olqer.forward(h(X), P, w_bits=w_bits)) <= 1.0
    for _ in range(4):
        assert torch.equal(L.linear(X, Pg, ws), Y)
    Pg.release()
