"""Calls that do the same work give the same bits, whatever else their launches carry.

The low-rank intermediate T is a sum over K that a launch of kernel 1 may split; how it is split depends on the layer and
the row count alone, so a forward, its two stages called one by one, every candidate of a clip search and every chunk of
a host-buffer forward add it up in the same order.
"""
import pytest
import torch

import paper_2605_27003_b200 as w4
from paper_2605_27003_b200 import build as pkg_build
from workloads import generator as gen

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# Rows on both sides of each edge of the split rule, and between them.
ROWS = [300, 448, 449, 700, 1024, 1025, 1560, 2300, 4352, 4353]
K, N, R = 2048, 1024, 64


@pytest.fixture(scope="module")
def setup():
    pkg_build.build()
    w4.load_library()
    layer = gen.make_layer_direct(K, N, R, seed=11).to(DEV)
    ctx = w4.Context(0, max(ROWS), K, R)
    L = w4.Layer(ctx, [layer], num_bins=1)
    x = gen.make_activations(max(ROWS), K, seed=12).to(DEV)
    yield ctx, L, layer, x, torch.full((1, 1, 1), 0.85, device=DEV)
    L.close()
    ctx.close()


@pytest.mark.parametrize("M", ROWS)
def test_a_forward_equals_its_two_stages(setup, M):
    ctx, L, _, x, clip = setup
    y = L.forward(x[:M], 0, 0, clip)
    staged = torch.empty_like(y)
    w4.w4a4_quantize_activations(L.ptr, x[:M], M, 0, 0, clip)
    w4.w4a4_gemm_from_workspace(L.ptr, M, 0, staged)
    assert torch.equal(y, staged)
    ctx.check()


@pytest.mark.parametrize("M", [700, 1560])
def test_every_candidate_of_a_search_is_scored_alike(setup, M):
    # The same ratio three times: the errors differ by the order of FP64 atomic sums alone (at most M * N terms of one sign).
    _, L, layer, x, _ = setup
    yref = gen.reference_output(x[:M].cpu(), layer.to("cpu")).to(DEV)
    table = torch.full((1, 1, 1), 1.0, device=DEV)
    _, errs = w4.w4a4_clip_search(L.ptr, [x[:M]], [yref], M, 0, 0, [0.85, 0.85, 0.85], table)
    assert max(errs) - min(errs) <= M * N * 2.0 ** -53 * max(errs)


@pytest.mark.parametrize("M", [700, 1560])
def test_every_chunk_of_a_host_forward_is_computed_alike(M):
    pkg_build.build()
    w4.load_library()
    layer = gen.make_layer_direct(K, N, R, seed=11).to(DEV)
    ctx = w4.Context(0, 3 * M, K, R)
    L = w4.Layer(ctx, [layer], num_bins=1)
    w4.w4a4_ctx_enable_host_io(ctx.ptr, M, N)
    x = gen.make_activations(M, K, seed=12)
    x3 = torch.cat([x, x, x]).pin_memory()
    y3 = torch.empty(3 * M, N, dtype=torch.bfloat16).pin_memory()
    clip = torch.full((1, 1, 1), 0.85, device=DEV)
    w4.w4a4_linear_forward_host(L.ptr, x3, 3 * M, 0, 0, clip, y3)
    torch.cuda.synchronize()
    assert torch.equal(y3[:M], y3[M:2 * M]) and torch.equal(y3[:M], y3[2 * M:])
    L.close()
    ctx.close()
