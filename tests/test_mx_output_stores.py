"""The MXFP4 GEMM's output by TMA stores: all of Y and nothing outside it, at ragged rows and at columns that half fill the last tile,
in its single-CTA form, as CTA pairs with several tiles each, and with the fused activation."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_27003_b200", "csrc")
SHIM = '#include "mx_gemm_plan.h"\nextern "C" int pairs(int m, int n, int sms) { return w4a4::mx_gemm_pairs(m, n, sms, false); }\n'


@pytest.fixture(scope="module")
def pairs(tmp_path_factory):
    d = tmp_path_factory.mktemp("mx_plan")
    src, lib = d / "plan.cpp", d / "plan.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(str(lib)).pairs


def shape(form, sms):
    """(M, N) that take the form on a device with that many SMs, with a tile of 33 rows or less at the end."""
    if form == "one row tile":
        return 97, 384                                        # N = 128 mod 256
    if form == "single CTAs, a tile each":
        return 300, 640
    if form == "single CTAs, more than a tile for some":
        m, n = next((m, n) for n in range(20, 3, -1) for m in range(3, sms) if sms < m * n <= sms + sms // 8)
        return 128 * (m - 1) + 4, 256 * n
    if form == "pairs, the last one with one row tile":
        return 128 * 12 + 33, 256 * (2 * (sms // 2) // 7)     # one wave of pairs, two of single CTAs
    assert form == "pairs, three tiles each and more"
    return 128 * 24 + 33, 256 * (-(-3 * (sms // 2) // 13)) + 128


# K is too short to be split: at least three stages of 256 would go to each CTA of a cluster.
@pytest.mark.parametrize("form,K,r,gelu,paired", [
    ("one row tile", 256, 0, False, False),
    ("single CTAs, a tile each", 512, 16, True, False),
    ("single CTAs, more than a tile for some", 256, 32, False, False),
    ("pairs, the last one with one row tile", 256, 64, True, True),
    ("pairs, three tiles each and more", 512, 16, False, True),
])
def test_outputs_stay_inside_y(pairs, form, K, r, gelu, paired):
    import paper_2605_27003_b200 as w4
    from test_gpu_parity import guarded
    from test_mx_gpu_parity import bits, mx_inputs
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M, N = shape(form, sms)
    tiles_m, tiles_n = -(-M // 128), -(-N // 256)
    assert bool(pairs(tiles_m, tiles_n, sms)) == paired
    x, layer = mx_inputs(M, K, N, r, seed=M, bias=True)
    ctx = w4.Context(0, M, K, r)
    lay = w4.MxLayer(ctx, [layer.to(DEV)], num_bins=1, output_activation=w4.ACT_GELU_TANH if gelu else w4.ACT_NONE)
    xd, clip = x.to(DEV), torch.full((1, 1, 1), 0.9, dtype=torch.float32, device=DEV)
    outputs = []
    for _ in range(2):
        buf, y = guarded((M, N), torch.bfloat16, float("nan"))   # what is not stored stays NaN
        w4.w4a4_mx_linear_forward(lay.ptr, xd, M, 0, 0, clip, y)
        torch.cuda.synchronize()
        ctx.check()
        assert int(torch.isnan(buf).sum()) == (buf.shape[0] - M) * N and not bool(torch.isnan(y).any())
        outputs.append(y)
    assert torch.equal(outputs[0], outputs[1])
    # A row of every 32-row block that a warp stores, all columns; the first and the last row.
    rows = np.unique(np.concatenate([[0, M - 1], (np.arange(0, M, 32) + (7 * np.arange(-(-M // 32))) % 32).clip(0, M - 1)]))
    ref = oracle.mx_forward_rows(bits(x), rows.astype(np.int32), layer.lam.numpy(), 0.9, None if r == 0 else bits(layer.L1),
                                 None if r == 0 else bits(layer.L2), layer.wcodes.numpy(), layer.wexps.numpy(), layer.bias.numpy())["Y64"]
    # The layer's tolerance; through the activation, whose slope is at most 1.13, that much more.
    bound = (1.13 if gelu else 1.0) * (2.0 ** -7 * np.abs(ref) + 1e-3 * float(np.sqrt(np.mean(ref ** 2))))
    got = outputs[0][torch.from_numpy(rows).to(DEV)].double().cpu().numpy()
    assert np.all(np.abs(got - (oracle.gelu_tanh(ref) if gelu else ref)) <= bound)
    lay.close()
    ctx.close()
