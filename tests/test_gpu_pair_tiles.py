"""Tile widths of the pair GEMM: batches of more than 128 rows whose tiles are 256, 192 or 128 columns wide.

Widths of 192 columns begin inside packed tiles of 128, so columns, their exponents and their blocks of B_q come from two of them;
N ends inside a tile, inside a half and right behind one.
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


@pytest.mark.parametrize("M,K,N,k,w_bits", [
    (300, 320, 4104, 40, 4),        # 34 tiles of 256: 128 wide (66)
    (300, 192, 7056, 16, 4),        # 56 tiles of 256: 192 wide (74), the last one 144
    (513, 208, 4616, 72, 4),        # three row tiles: 57 of 256, 75 of 192: 256 wide
    (513, 208, 4616, 0, 2),
    (300, 256, 6920, 256, 2),       # 192 wide, crumbs, rank blocks that straddle packed tiles
    (201, 256, 10992, 20, 4),       # 192 wide, one row tile
], ids=lambda v: str(v))
def test_tile_widths_against_the_oracle(M, K, N, k, w_bits):
    spec = gen.LayerSpec("width", M=M, K=K, N=N, k=k, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=911)
    W = gen.make_weight(spec)
    A, B = gen.make_random_factors(spec) if k else (None, None)
    cfg = L.default_config()
    cfg.w_bits = w_bits
    P = olqer.prepare_weights(W, A, B, w_bits=w_bits)
    Pg = L.prepare_weights(_t(W), *((_t(A), _t(B)) if k else (None, None)), cfg)
    X = gen.make_activations(spec)
    ref = olqer.forward(X, P, w_bits=w_bits)
    ws = L.new_workspace(M, Pg)
    Xg = _t(X)
    Y = L.linear(Xg, Pg, ws)
    assert L.poll_status(ws) == 0
    assert worst_ratio(Y.cpu().numpy(), ref) <= 1.0
    if M > 256:                                        # (no K ranges there: the same fp32 values whatever the type of Y)
        assert torch.equal(L.linear_ex(Xg, Pg, ws, out_dtype=torch.bfloat16), Y.bfloat16())
        if N % 16 == 0:
            assert torch.equal(L.linear_ex(Xg, Pg, ws, out_dtype=L.MXINT8), L.to_mxint8(*L.quantize_activations(Y, cfg)))
    else:
        got = L.linear_ex(Xg, Pg, ws, out_dtype=torch.bfloat16).float()
        assert torch.all((got - Y).abs() <= Y.abs() * 2.0 ** -8 + torch.from_numpy(ref.tol).to(DEV))   # a bf16 unit and the tolerance
    Pg.release()
