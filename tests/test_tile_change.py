"""The INT4 GEMM's tile change: several tiles per CTA with every parity of TMEM slot uses per tile (groups and the low-rank
entry), the output's TMA stores at ragged row counts and exact sub-tile boundaries."""
import numpy as np
import pytest
import torch

from workloads import generator as gen

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N = 2560   # 20 column tiles: with 25 row blocks more than three tiles per CTA


@pytest.mark.parametrize("K,r", [(64, 0), (64, 16), (128, 0), (128, 32), (192, 0), (192, 16), (320, 96), (704, 64)])
@pytest.mark.parametrize("M", [3072 + 33, 3072 + 96])
def test_several_tiles_per_cta(K, r, M):
    import paper_2605_27003_b200 as w4
    from test_gpu_parity import guarded, guards_intact, oracle_rows, y_within_tolerance
    x = gen.make_activations(M, K, outlier_idx=gen.outlier_channels(K, 0, 3, count=2), outlier_gain=20.0, seed=3)
    layer = gen.make_layer_svd(K, N, r, x[:1024], seed=4, bias_std=0.01)
    ctx = w4.Context(0, M, K, r)
    lay = w4.Layer(ctx, [layer.to(DEV)], num_bins=1)
    xd, clip = x.to(DEV), torch.full((1, 1, 1), 0.9, dtype=torch.float32, device=DEV)
    y_buf, y = guarded((M, N), torch.bfloat16, 1234.0)
    w4.w4a4_linear_forward(lay.ptr, xd, M, 0, 0, clip, y)
    torch.cuda.synchronize()
    ctx.check()
    assert guards_intact(y_buf, 1234.0)
    rows = np.array([0, 31, 32, 127, 128, 1000, 2047, 3071, 3072, M - 2, M - 1])
    worst, _ = y_within_tolerance(y[torch.from_numpy(rows).to(DEV)], oracle_rows(x[rows], layer, 0.9)["Y64"])
    assert worst <= 1.0
    # A tile whose epilogue lags (it stores its partial sums) must not let any other role run into an older phase.
    bm, bn = w4.w4a4_tile_shape()
    P = torch.empty(bm, K // 64, bn, dtype=torch.int32, device=DEV)
    for m0, n0 in ((0, 0), (1536, 1280), (3072, N - 128)):
        y2_buf, y2 = guarded((M, N), torch.bfloat16, 1234.0)
        w4.w4a4_debug_partials(lay.ptr, xd, M, 0, 0, clip, y2, m0, n0, P)
        torch.cuda.synchronize()
        ctx.check()
        assert torch.equal(y, y2) and guards_intact(y2_buf, 1234.0)
    lay.close()
    ctx.close()
