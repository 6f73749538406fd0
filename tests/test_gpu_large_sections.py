"""A layer whose packed weights take more than 4 GiB: offsets into them need more than 32 bits (few rows only; larger batches
take the same section by 64-bit offsets in the GEMMs)."""
import numpy as np
import pytest
import torch

import lqer_inputs as gen
import paper_2402_02446_b200 as L
from oracle import lqer as olqer
from helpers import worst_ratio

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
K, N, RANK = 16384, 466944, 16                  # 3648 column tiles of 256 slabs of 4608 bytes: 8 tiles of them behind 4 GiB


@pytest.fixture(scope="module")
def layer():
    if torch.cuda.mem_get_info()[0] < 48 << 30:
        pytest.skip("the unpacked weights alone take 31 GB")
    g = torch.Generator(device=DEV)
    g.manual_seed(931)
    W = torch.empty((K, N), device=DEV)
    for rows in W.split(1024):
        rows.normal_(0.0, 0.02, generator=g)
    A = torch.randn((K, RANK), generator=g, device=DEV) / K ** 0.5
    B = torch.randn((RANK, N), generator=g, device=DEV) * 0.01
    # the first columns, two of the last tiles (behind 4 GiB) and one in between
    cols = torch.cat([torch.arange(0, 16), torch.arange(N // 2, N // 2 + 8), torch.arange(N - 200, N - 184), torch.arange(N - 16, N)]).to(DEV)
    P = olqer.prepare_weights(W[:, cols].cpu().numpy(), A.cpu().numpy(), B[:, cols].cpu().numpy())
    Pg = L.prepare_weights(W, A, B)
    torch.cuda.synchronize()
    del W
    torch.cuda.empty_cache()
    yield P, Pg, cols
    Pg.release()
    del Pg
    torch.cuda.empty_cache()


@pytest.mark.parametrize("M,n", [(1, 1), (3, 1), (4, 1), (8, 1), (2, 2), (5, 2), (4, 6)])
def test_columns_beyond_four_gigabytes(layer, M, n):
    P, Pg, cols = layer
    spec = gen.LayerSpec("large", M=M, K=K, N=N, k=RANK, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=932)
    Xs = [gen.make_activations(spec, M=M) + np.float32(0.25 * i) for i in range(n)]
    xs = [torch.from_numpy(x).to(DEV) for x in Xs]
    Ys = [torch.full((M, N), float("nan"), device=DEV) for _ in range(n)]
    calls = L.make_calls([(x, Pg, y) for x, y in zip(xs, Ys)])
    ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=DEV)
    L.linear_batched(calls, ws)
    assert L.poll_status(ws) == 0
    for x, y in zip(Xs, Ys):
        assert worst_ratio(y[:, cols].cpu().numpy(), olqer.forward(x, P)) <= 1.0
