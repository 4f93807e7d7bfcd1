"""The MXFP4 GEMM's output by TMA stores: nothing outside Y, at ragged rows and at columns that half fill the last tile, in its
single-CTA form, as CTA pairs with several tiles each, and with the fused activation."""
import numpy as np
import pytest
import torch

import oracle
from workloads import generator as gen

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("M,K,N,r,gelu", [
    (97, 256, 384, 0, False),      # one row tile, N = 128 mod 256
    (300, 512, 640, 16, True),     # single CTAs, K too short to be split
    (900, 256, 5120, 32, False),   # a single CTA per tile, more than one tile each
    (1569, 256, 5120, 64, True),   # CTA pairs, the last pair with one row tile of 33 rows
    (3105, 512, 2688, 16, False),  # several tiles per pair, N = 128 mod 256
])
def test_outputs_stay_inside_y(M, K, N, r, gelu):
    import paper_2605_27003_b200 as w4
    from test_gpu_parity import guarded, guards_intact
    from test_mx_gpu_parity import bits, mx_inputs
    x, layer = mx_inputs(M, K, N, r, seed=M, bias=True)
    ctx = w4.Context(0, M, K, r)
    lay = w4.MxLayer(ctx, [layer.to(DEV)], num_bins=1, output_activation=w4.ACT_GELU_TANH if gelu else w4.ACT_NONE)
    xd, clip = x.to(DEV), torch.full((1, 1, 1), 0.9, dtype=torch.float32, device=DEV)
    buf, y = guarded((M, N), torch.bfloat16, 1234.0)
    for _ in range(2):
        w4.w4a4_mx_linear_forward(lay.ptr, xd, M, 0, 0, clip, y)
    torch.cuda.synchronize()
    ctx.check()
    assert guards_intact(buf, 1234.0)
    rows = np.unique(np.array([0, 31, 32, M // 2, M - 33, M - 32, M - 2, M - 1]).clip(0, M - 1))
    ref = oracle.mx_forward_rows(bits(x), rows.astype(np.int32), layer.lam.numpy(), 0.9, None if r == 0 else bits(layer.L1),
                                 None if r == 0 else bits(layer.L2), layer.wcodes.numpy(), layer.wexps.numpy(), layer.bias.numpy())["Y64"]
    # The layer's tolerance; through the activation, whose slope is at most 1.13, that much more.
    bound = (1.13 if gelu else 1.0) * (2.0 ** -7 * np.abs(ref) + 1e-3 * float(np.sqrt(np.mean(ref ** 2))))
    got = y[torch.from_numpy(rows).to(DEV)].double().cpu().numpy()
    assert np.all(np.abs(got - (oracle.gelu_tanh(ref) if gelu else ref)) <= bound)
    lay.close()
    ctx.close()
