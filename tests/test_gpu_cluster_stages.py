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
        Y = L.linear(Xg, Pg, ws)
        again = L.linear(Xg, Pg, ws)
        assert L.poll_status(ws) == 0
        assert torch.equal(Y, again)
        assert worst_ratio(Y.cpu().numpy(), ref) <= 1.0, M
    Pg.release()
