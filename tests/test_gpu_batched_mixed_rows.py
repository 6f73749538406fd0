"""Batches whose calls differ in their rows: a stretch of one- to four-row calls has its activations computed ahead into the
workspace, and a run in its middle that another kernel could take must not lose what the rest of the stretch still reads."""
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


@pytest.mark.parametrize("rows", [
    [1] * 2 + [3] * 3 + [1] * 14,            # three neighbours that fit one launch of the cluster kernel
    [2] * 2 + [4] * 7 + [2] * 10,            # seven that the launches of many small batches would take
    [1] * 17 + [4] * 2 + [1] * 3 + [3] * 4 + [2] * 5,
], ids=["three-of-3", "seven-of-4", "several"])
def test_runs_in_the_middle_of_a_stretch(rows):
    # layers so small that no launch fills the GPU: the next run may then choose its kernel anew
    specs = [gen.LayerSpec(f"mix{i}", M=4, K=256, N=256, k=16, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=921 + i)
             for i in range(3)]
    layers = []
    for s in specs:
        W = gen.make_weight(s)
        A, B = gen.make_random_factors(s)
        layers.append((olqer.prepare_weights(W, A, B), L.prepare_weights(_t(W), _t(A), _t(B))))
    Xs = [gen.make_activations(specs[i % 3], M=m) + np.float32(0.125 * i) for i, m in enumerate(rows)]
    xs = [_t(x) for x in Xs]
    Ys = [torch.full((m, 256), float("nan"), device=DEV) for m in rows]
    calls = L.make_calls([(x, layers[i % 3][1], y) for i, (x, y) in enumerate(zip(xs, Ys))])
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    for _ in range(2):
        L.linear_batched(calls, ws)
        assert L.poll_status(ws) == 0
        for i, (x, y) in enumerate(zip(Xs, Ys)):
            assert worst_ratio(y.cpu().numpy(), olqer.forward(x, layers[i % 3][0])) <= 1.0, i
            y.fill_(float("nan"))
    for _, Pg in layers:
        Pg.release()
