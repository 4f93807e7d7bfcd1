"""The calls whose speed matters to a user of this package, as seeded cases: the quantized linears of a video DiT at
its latent sizes, on both 4-bit grids, and the offline steps that prepare them (clip-ratio search, GPTQ).

`listed()` names the fixed cases, `draw()` gives further ones of the same ranges; `prepare()` builds what a program
holds before the call (activations, packed layer, context, clip table), `run()` is one call through the public entry
points.  Shapes: hidden width 5120, FFN width 13824, 32760 tokens (21 x 30 x 52 latent), 1560 tokens (one latent
frame), a 512-wide toy layer, and generic ragged ones.
"""
import math
from types import SimpleNamespace

import torch

import paper_2605_27003_b200 as w4

CANDIDATES = (0.5, 0.6, 0.7, 0.8, 0.9, 1.0)   # ratios a clip search tries
SEARCH_SAMPLES = 2                            # calibration samples per search
BINS = 8                                      # timestep bins of the clip table


def _linear(name, grid, M, K, N, r, gelu=False, dist="normal", experts=1):
    return dict(name=name, kind=grid, M=M, K=K, N=N, r=r, gelu=gelu, dist=dist, experts=experts)


def listed():
    return [
        # The toy layer of the unit tests and of a first trial: latency and launches are all there is.
        _linear("int4_tiny", "int4", 256, 512, 512, 16),
        # One latent frame (previews, short clips, the low end of the shape sweep), widest single-layer rank.
        _linear("int4_frame", "int4", 1560, 5120, 5120, 64),
        # q, k and v of one block packed as a layer of joint rank 96, ragged token count.
        _linear("int4_qkv_ragged", "int4", 4097, 5120, 15360, 96),
        # Attention projection of a denoising step, both experts' weights resident.
        _linear("int4_attn_proj", "int4", 32760, 5120, 5120, 32, experts=2),
        # FFN of the same step: up-projection with the fused GELU, down-projection of GELU-shaped activations.
        _linear("int4_ffn_up", "int4", 32760, 5120, 13824, 32, gelu=True),
        _linear("int4_ffn_down", "int4", 32760, 13824, 5120, 32, dist="gelu"),
        # A handful of rows through a full-size layer (conditioning tokens, batch-of-one modulation), no low-rank pair.
        _linear("mx_rows", "mx", 100, 5120, 5120, 0),
        # The MXFP4 grid at one latent frame and at the full latent.
        _linear("mx_frame", "mx", 1560, 5120, 13824, 32),
        _linear("mx_attn_proj", "mx", 32760, 5120, 5120, 32),
        # The whole FFN of a step on the MXFP4 grid in one call.
        dict(name="mx_ffn", kind="mx_ffn", M=32760, K=5120, H=13824, N=5120, r=32),
        # Calibration: the clip-ratio search of one (expert, layer, bin) on one latent frame per sample.
        dict(name="clip_search", kind="clip", M=1560, K=5120, N=5120, r=32),
        # Calibration: GPTQ of one layer's residual weights from 2048 calibration tokens.
        dict(name="gptq", kind="gptq", K=5120, N=5120, M_cal=2048, mx=False),
    ]


_MAX_MKN = 32760 * 5120 * 13824


def _log_uniform(rng, lo, hi, multiple=1):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple
    return min(max(v, -(-lo // multiple) * multiple), hi // multiple * multiple)


def draw(rng):
    kind = rng.choices(("int4", "mx", "mx_ffn", "clip", "gptq"), weights=(6, 3, 1, 1, 1))[0]
    if kind == "gptq":
        K, N = _log_uniform(rng, 512, 5120, 64), _log_uniform(rng, 128, 5120, 64)
        return dict(kind=kind, K=K, N=N, M_cal=_log_uniform(rng, 256, 2048), mx=rng.random() < 0.5)
    if kind == "mx_ffn":
        K, H, N = _log_uniform(rng, 512, 5120, 256), _log_uniform(rng, 1024, 13824, 256), _log_uniform(rng, 512, 5120, 256)
        return dict(kind=kind, M=_log_uniform(rng, 129, 32760), K=K, H=H, N=N, r=rng.choice((16, 32, 64)))
    K = _log_uniform(rng, 512, 13824, 256 if kind == "mx" else 64)
    N = _log_uniform(rng, 512, 15360, 128)
    if kind == "clip":
        most = min(8192, _MAX_MKN // (K * N * len(CANDIDATES) * SEARCH_SAMPLES))
        return dict(kind=kind, M=_log_uniform(rng, 200, most), K=K, N=N, r=rng.choice((0, 16, 32, 64)))
    M = _log_uniform(rng, 1, min(75600, _MAX_MKN // (K * N)))
    r = rng.choice((0, 16, 32, 64, 96) if kind == "int4" else (0, 16, 32, 64))
    return dict(kind=kind, M=M, K=K, N=N, r=r, gelu=rng.random() < 0.25, dist=rng.choice(("normal", "gelu")), experts=1)


# --------------------------------------------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _activations(M, K, g, dist, sigma):
    """BF16 tokens: Gaussian (or GELU of a Gaussian, the input of an FFN's second linear), 1 % of the channels x 50."""
    x = torch.randn(M, K, generator=g, device="cuda", dtype=torch.bfloat16)
    if dist == "gelu":
        x = torch.nn.functional.gelu(x)
    gain = torch.full((K,), sigma, device="cuda")
    gain[torch.randperm(K, generator=g, device="cuda")[: max(1, K // 100)]] *= 50.0
    return x.mul_(gain.to(torch.bfloat16))


def _constants(K, N, r, g, grid):
    """One expert's constants as calibration hands them over: smoothing vector, low-rank pair, bias, 4-bit residual."""
    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    c = SimpleNamespace(K=K, N=N, r=r, lam=torch.exp(0.5 * normal(K)), bias=0.01 * normal(N), L1=None, L2=None)
    if r > 0:
        c.L1, c.L2 = (0.05 * normal(K, r)).to(torch.bfloat16), (0.05 * normal(r, N)).to(torch.bfloat16)
    if grid == "mx":
        c.wcodes = torch.randint(0, 16, (K, N), generator=g, device="cuda", dtype=torch.uint8)
        c.wexps = torch.randint(118, 122, (K // 32, N), generator=g, device="cuda", dtype=torch.uint8)
    else:
        c.qweight = torch.round(2.5 * normal(K, N)).clamp_(-8, 7).to(torch.int8)
        c.wscale = 2e-3 * torch.exp(math.log(10.0) * torch.rand(K // 64, N, generator=g, device="cuda"))
    return c


def _clip_table(experts, layers, g):
    return 0.6 + 0.4 * torch.rand(experts, layers, BINS, generator=g, device="cuda")


def _full_precision_output(x, c):
    """The BF16 output a calibration run records for Eq. 10: X W + b, W = diag(1 / lambda) (L1 L2 + codes * scales)."""
    w = c.qweight.float().view(-1, 64, c.N).mul_(c.wscale.unsqueeze(1)).view(c.K, c.N)
    if c.r > 0:
        w += c.L1.float() @ c.L2.float()
    w /= c.lam.unsqueeze(1)
    return (x.float() @ w + c.bias).to(torch.bfloat16)


def prepare(case, seed):
    kind, g = case["kind"], _generator(seed)
    s = SimpleNamespace(kind=kind)
    if kind == "gptq":
        K, N, M = case["K"], case["N"], case["M_cal"]
        # Correlated calibration activations (shared directions on independent noise, a few large channels).
        x = torch.randn(M, K, generator=g, device="cuda")
        x += 0.8 * torch.randn(M, 8, generator=g, device="cuda") @ torch.randn(8, K, generator=g, device="cuda")
        x[:, torch.randperm(K, generator=g, device="cuda")[: max(2, K // 128)]] *= 6.0
        s.mx, s.xhat = case["mx"], x.to(torch.bfloat16)
        s.R = 0.02 * torch.randn(K, N, generator=g, device="cuda")
        s.codes = torch.empty(K, N, device="cuda", dtype=torch.uint8 if s.mx else torch.int8)
        s.scales = torch.empty(K // (32 if s.mx else 64), N, device="cuda", dtype=torch.uint8 if s.mx else torch.float32)
        s.workspace = torch.empty(w4.w4a4_gptq_workspace_bytes(K, N, M), device="cuda", dtype=torch.uint8)
        return s
    M, K, N, r = case["M"], case["K"], case["N"], case["r"]
    s.M, s.bin = M, seed % BINS
    sigma = 2.0 * 0.8 ** s.bin     # activations shrink over the timesteps
    s.Y = torch.empty(M, N, device="cuda", dtype=torch.bfloat16)
    if kind == "clip":
        s.ctx = w4.Context(0, M, K, r)
        c = _constants(K, N, r, g, "int4")
        s.layer = w4.Layer(s.ctx, [c], num_bins=BINS)
        s.X = [_activations(M, K, g, "normal", sigma) for _ in range(SEARCH_SAMPLES)]
        s.Yref = [_full_precision_output(x, c) for x in s.X]
        s.clip = _clip_table(1, 1, g)
        return s
    if kind == "mx_ffn":
        H = case["H"]
        s.ctx = w4.Context(0, M, max(K, H), r)
        s.up = w4.MxLayer(s.ctx, [_constants(K, H, r, g, "mx")], num_bins=BINS, num_layers=2, layer_id=0,
                          output_activation=w4.ACT_GELU_TANH)
        s.down = w4.MxLayer(s.ctx, [_constants(H, N, r, g, "mx")], num_bins=BINS, num_layers=2, layer_id=1)
        s.X, s.clip = _activations(M, K, g, "normal", sigma), _clip_table(1, 2, g)
        return s
    s.ctx = w4.Context(0, M, K, r)
    s.expert = case["experts"] - 1
    make = w4.MxLayer if kind == "mx" else w4.Layer
    s.layer = make(s.ctx, [_constants(K, N, r, g, kind) for _ in range(case["experts"])], num_bins=BINS,
                   output_activation=w4.ACT_GELU_TANH if case["gelu"] else w4.ACT_NONE)
    s.X, s.clip = _activations(M, K, g, case["dist"], sigma), _clip_table(case["experts"], 1, g)
    return s


# ------------------------------------------------------------------------------------------------------- one pass
def run(s):
    if s.kind == "gptq":
        fn = w4.w4a4_mx_gptq_quantize if s.mx else w4.w4a4_gptq_quantize
        fn(s.R, s.codes, s.scales, Xhat=s.xhat, workspace=s.workspace)
        return s.codes, s.scales
    if s.kind == "clip":
        best, errors = w4.w4a4_clip_search(s.layer.ptr, s.X, s.Yref, s.M, 0, s.bin, CANDIDATES, s.clip)
        return best, errors, s.clip
    if s.kind == "mx_ffn":
        w4.w4a4_mx_ffn_forward(s.up.ptr, s.down.ptr, s.X, s.M, 0, s.bin, s.clip, s.Y)
        return s.Y
    return s.layer.forward(s.X, s.expert, s.bin, s.clip, s.Y)


def _linear_work(M, K, N, r, mx, passes=1):
    """X read and Y written once, the constants once: 4-bit codes, their scales, low-rank pair, smoothing, bias."""
    scales = K // 32 * N if mx else 4 * (K // 64) * N
    constants = K * N // 2 + scales + 2 * r * (K + N) + 4 * (K + N)
    return dict(bytes=2 * M * (K + N) + constants, flops=passes * 2 * M * (K * N + r * (K + N)))


def work(case):
    kind = case["kind"]
    if kind == "gptq":
        K, N, M = case["K"], case["N"], case["M_cal"]
        # statistic (upper triangle), factorization and triangular inverse, the sweep's updates: FP64
        flops = M * K * K + 2 * K ** 3 // 3 + K * K * N
        out = K * N + (K // 32 * N if case["mx"] else 4 * (K // 64) * N)
        return dict(bytes=2 * M * K + 4 * K * N + out, flops=flops)
    M, K, N, r = case["M"], case["K"], case["N"], case["r"]
    if kind == "mx_ffn":
        H = case["H"]
        up, down = _linear_work(M, K, H, r, True), _linear_work(M, H, N, r, True)
        return dict(bytes=up["bytes"] + down["bytes"] - 4 * M * H, flops=up["flops"] + down["flops"])
    if kind == "clip":
        once = _linear_work(M, K, N, r, False, passes=SEARCH_SAMPLES * len(CANDIDATES))
        once["bytes"] += (SEARCH_SAMPLES - 1) * 2 * M * (K + N)
        return once
    return _linear_work(M, K, N, r, kind == "mx")


def tolerance(case):
    """About four times what the path showed against itself in FP64 on the same 4-bit codes (outputs rounded to BF16)."""
    kind = case["kind"]
    if kind == "gptq":
        # None of the whole values differed; a weight within 1e-10 of a rounding boundary may still take the other code
        # under another FP64 summation order, and its output channel then follows another valid course: one channel of 512.
        return {"rel": 2e-3, "max": 0.5, "differ": 2e-3}
    if kind == "clip":
        return {"rel": 4e-6, "max": 4e-6}       # sums over millions of squared errors: 8.6e-7 seen
    if kind == "mx_ffn":
        # 1.8e-4 and 0.013 seen: a hidden value that rounds the other way moves its 4-bit code
        return {"rel": 7e-4, "max": 0.05}
    return {"rel": 5e-4, "max": 0.016}          # 1.2e-4 and one BF16 step (0.0078) seen
