"""Separate contexts are independent: host threads that drive one each get the results they would get alone.

Two threads, each with its own context, layer and stream, run the same instantiation of kernel 1 with row counts whose
launches differ (CTA size, shared memory).  Outputs of every call have to be those of a run without the other thread.
"""
import os
import subprocess
import sys
import threading

import pytest
import torch

import paper_2605_27003_b200 as w4
from paper_2605_27003_b200 import build as pkg_build
from workloads import generator as gen

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("grid", ["int4", "mx"])
def test_threads_with_contexts_of_their_own_do_not_meet(grid):
    pkg_build.build()
    w4.load_library()
    K, N, r, calls = 2048, 256, 64, 1500
    clip = torch.full((1, 1, 1), 0.9, device=DEV)
    layer = (gen.make_layer_mx_direct if grid == "mx" else gen.make_layer_direct)(K, N, r, seed=1).to(DEV)
    jobs = []
    for M in (200, 448):
        ctx = w4.Context(0, M, K, r)
        L = (w4.MxLayer if grid == "mx" else w4.Layer)(ctx, [layer], num_bins=1)
        x = gen.make_activations(M, K, seed=M).to(DEV)
        y = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
        alone = torch.empty_like(y)
        L.forward(x, 0, 0, clip, alone)
        jobs.append((ctx, L, x, y, alone, torch.cuda.Stream()))
    torch.cuda.synchronize()
    start, failures = threading.Barrier(len(jobs)), []

    def work(ctx, L, x, y, alone, stream):
        try:
            with torch.cuda.stream(stream):
                start.wait()
                for _ in range(calls):
                    L.forward(x, 0, 0, clip, y, stream)
                stream.synchronize()
            if not torch.equal(y, alone):
                failures.append(f"{x.shape[0]} rows: other outputs than alone")
        except Exception as e:
            failures.append(f"{x.shape[0]} rows: {e}")

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
    for ctx, L, *_ in jobs:
        ctx.check()
        L.close()
        ctx.close()


FIRST_CALL = """
import torch, paper_2605_27003_b200 as w4
from workloads import generator as gen
mx, K, N, r, M = {mx}, 2048, 256, 64, 1
layer = (gen.make_layer_mx_direct if mx else gen.make_layer_direct)(K, N, r, seed=1).to("cuda:0")
ctx = w4.Context(0, M, K, r)
L = (w4.MxLayer if mx else w4.Layer)(ctx, [layer], num_bins=1)
L.forward(gen.make_activations(M, K, seed=2).to("cuda:0"), 0, 0, torch.full((1, 1, 1), 0.9, device="cuda:0"))
torch.cuda.synchronize()
ctx.check()
"""


@pytest.mark.parametrize("mx", [False, True])
def test_the_first_call_of_a_process_needs_no_larger_one_before_it(mx):
    # This plan's dynamic shared memory is 48 KiB exactly: with the kernel's static part it is more than a launch may take
    # unless the kernel's limit has been raised.
    pkg_build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", FIRST_CALL.format(mx=mx)], cwd=root, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
