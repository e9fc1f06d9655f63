"""The work a user of this library has it do, as measurable cases.

Every case goes through the public binding (`paper_2602_01410_b200.api`) the way a training program calls it: inputs, output
buffers, statistics buffers and the workspace exist before the call and are kept from step to step.  Shapes and tags are those
of the configurations in `paper_2602_01410_b200/workloads.py` (single 512 linear, Llama-like 1B / 3B / 7B / 70B linears); tensors
are drawn on the device with that module's distributions (activations with outlier channels, weights of standard deviation 0.02,
output gradients with a per-token log-normal factor).

Kinds of case
  linear   forward and both gradients of one linear layer under a precision triple, every tensor read once, statistics on
           (pow2 = 0: the paper's scale rule; 1 / 2: power-of-two scales on 128- / 32-long tiles; sr: stochastic rounding of FP4 dY)
  tagged   the three separate calls, for layers in which a GEMM keeps BF16 (statistics on)
  nvfp4    forward and both gradients under the two-level block-scaling option
  forward  a micro-batch against a weight that was quantized once for the optimizer step: quantize X, multiply
  stats    the collection step of the method: Frobenius norms of six tensors and the error norms of all options
  adamw    the optimizer sensitivity norm of one parameter tensor
"""
import math

import torch

from paper_2602_01410_b200 import api

BF16, FP8, FP4 = api.FMT_BF16, api.FMT_FP8_E4M3, api.FMT_FP4_E2M1
STATS_BYTES = 24   # one snip_stats_t: two float64 sums, a float32 maximum, padding


def _linear(name, M, K, N, fwd, dgrad, wgrad, pow2=0, sr=False):
    return {"name": name, "kind": "linear", "M": M, "K": K, "N": N, "fwd": fwd, "dgrad": dgrad, "wgrad": wgrad, "pow2": pow2, "sr": sr}


def listed():
    return [
        # the smallest call: one 512 x 512 linear over 512 tokens, fwd / dgrad FP8, wgrad FP4 (latency and launches count)
        _linear("single-512", 512, 512, 512, FP8, FP8, FP4),
        # grouped-query key / value projection of the 1B model: many tokens, a narrow output
        _linear("1b-kv", 8192, 2048, 256, FP8, FP4, FP8),
        # down projection of the 3B model: 8640 features end in a 64-wide tile; FP4 gradients rounded stochastically
        _linear("3b-down", 8192, 8640, 3200, FP4, FP8, FP4, sr=True),
        # fused query/key/value projection of the 7B model, all FP8
        _linear("7b-qkv-fp8", 16384, 4096, 12288, FP8, FP8, FP8),
        # gate projection of the 7B model, all FP4
        _linear("7b-gate-fp4", 16384, 4096, 11008, FP4, FP4, FP4),
        # the largest: down projection of the 70B model, mostly FP4
        _linear("70b-down", 8192, 28672, 8192, FP4, FP4, FP8),
        # output projection of the 7B model under the power-of-two scale option
        _linear("7b-o-pow2", 16384, 4096, 4096, FP8, FP8, FP4, pow2=1),
        # a gate projection of the 1B model with two of its three GEMMs kept in BF16 (tags are drawn per GEMM there)
        {"name": "1b-gate-tagged", "kind": "tagged", "M": 8192, "K": 2048, "N": 5632, "fwd": BF16, "dgrad": FP8, "wgrad": BF16},
        # gate projection of the 3B model under the two-level option, stochastic rounding of dY
        {"name": "3b-gate-nvfp4", "kind": "nvfp4", "M": 8192, "K": 3200, "N": 8640, "sr": True},
        # a micro-batch of 1024 tokens through a 7B output projection whose weight is already quantized
        {"name": "7b-o-microbatch", "kind": "forward", "M": 1024, "K": 4096, "N": 4096, "fmt": FP8},
        # the statistics collection of one 3B linear
        {"name": "3b-qkv-stats", "kind": "stats", "M": 8192, "K": 3200, "N": 9600},
        # the sensitivity norm of a 7B up-projection weight, bf16 gradients
        {"name": "7b-up-adamw", "kind": "adamw", "N": 11008, "K": 4096, "grad32": False},
    ]


def _dim(rng, lo, hi):
    """A multiple of 64 (odd multiples end in a 64-wide tile), spread over the logarithm of the range."""
    return 64 * max(1, round(math.exp(rng.uniform(math.log(lo / 64), math.log(hi / 64)))))


def _shape(rng, most, tokens=(512, 16384)):
    """Tokens, in-features and out-features of a linear whose M*N*K stays within `most`."""
    while True:
        M, K, N = _dim(rng, *tokens), _dim(rng, 256, 28672), _dim(rng, 256, 28672)
        if M * K * N <= most:
            return {"M": M, "K": K, "N": N}


def draw(rng):
    largest = 8192 * 28672 * 8192
    kind = rng.choices(["linear", "pow2", "tagged", "nvfp4", "forward", "stats", "adamw"], [6, 1, 1, 1, 1, 1, 1])[0]
    if kind in ("linear", "pow2"):
        f = [rng.choice([FP8, FP4]) for _ in range(3)]
        sr = FP4 in f[1:] and rng.random() < 0.5
        return {"kind": "linear", **_shape(rng, largest // 2), "fwd": f[0], "dgrad": f[1], "wgrad": f[2],
                "pow2": rng.choice([1, 2]) if kind == "pow2" else 0, "sr": sr}
    if kind == "tagged":
        f = [rng.choice([BF16, FP8, FP4]) for _ in range(3)]
        f[rng.randrange(3)] = BF16
        return {"kind": "tagged", **_shape(rng, largest // 4), "fwd": f[0], "dgrad": f[1], "wgrad": f[2]}
    if kind == "nvfp4":
        return {"kind": "nvfp4", **_shape(rng, largest // 2), "sr": rng.random() < 0.5}
    if kind == "forward":
        return {"kind": "forward", **_shape(rng, largest // 8, tokens=(256, 4096)), "fmt": rng.choice([FP8, FP4])}
    if kind == "stats":
        return {"kind": "stats", **_shape(rng, largest // 2)}
    return {"kind": "adamw", "N": _dim(rng, 256, 28672), "K": _dim(rng, 256, 8192), "grad32": rng.random() < 0.5}


# ---- inputs ----------------------------------------------------------------------------------------


def _normal(gen, rows, cols):
    return torch.randn(rows, cols, generator=gen, device="cuda", dtype=torch.float32)


def _x(gen, M, K):
    x = _normal(gen, M, K)
    x[:, torch.randperm(K, generator=gen, device="cuda")[: math.ceil(0.01 * K)]] *= 20.0
    return x.bfloat16()


def _w(gen, N, K):
    return (_normal(gen, N, K) * 0.02).bfloat16()


def _dy(gen, M, N):
    return (_normal(gen, M, N) * 1e-3 * _normal(gen, M, 1).exp()).bfloat16()


def _stats_views(raw):
    """The sums and the maximum of the snip_stats_t records in a byte buffer, as views of it."""
    rec = raw.view(-1, STATS_BYTES)
    return rec[:, :16].view(torch.float64), rec[:, 16:20].view(torch.float32)


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def _bf16(rows, cols):
    return torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda")


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, N, K = case["kind"], case["N"], case["K"]
    s = {"case": case}
    if kind == "adamw":
        g = _normal(gen, N, K) * 1e-3
        s["m"] = _normal(gen, N, K).mul_(3e-4).add_(g, alpha=0.1)
        s["v"] = _normal(gen, N, K).mul_(1e-3).square_().add_(g.square(), alpha=0.05)
        s["g"] = g if case["grad32"] else g.bfloat16()
        s["out"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        return s
    M = case["M"]
    s["x"], s["w"] = _x(gen, M, K), _w(gen, N, K)
    if kind == "forward":
        fmt = case["fmt"]
        codes, scales, _, _ = api.snip_quantize(s["w"], fmt, api.BLOCK_BLK)   # once per optimizer step
        s["wq"] = (codes, scales)
        s["w_op"] = api.make_qtensor(codes, scales, N, K, fmt, api.BLOCK_BLK)
        cb, sb, wb = api.snip_quantize_sizes(M, K, fmt, api.BLOCK_ROW, api.Q_STATS)
        s["codes"], s["scales"] = _bytes(cb).zero_(), torch.empty(sb // 4, dtype=torch.float32, device="cuda")   # FP4 codes may end in unused slack
        s["x_op"] = api.make_qtensor(s["codes"], s["scales"], M, K, fmt, api.BLOCK_ROW)
        s["stats"], s["qws"] = _bytes(STATS_BYTES), _bytes(wb)
        s["gws"] = _bytes(api.snip_workspace_size(api.OP_FWD, M, N, K, fmt, fmt)[0])
        s["sums"], s["amax"] = _stats_views(s["stats"])
        s["y"] = _bf16(M, N)
        return s
    s["dy"] = _dy(gen, M, N)
    if kind == "stats":
        s["y"], s["dx"] = _normal(gen, M, N).bfloat16(), (_normal(gen, M, K) * 1e-3).bfloat16()
        s["dw"] = (_normal(gen, N, K) * 1e-2).bfloat16()
        s["out"] = torch.zeros(24, dtype=torch.float64, device="cuda")
        s["ws"] = _bytes(api.snip_layer_stats_workspace(M, N, K))
        return s
    if kind == "nvfp4":
        # bounds of the three tensors, as the maxima an earlier step's statistics hold
        s["bounds"] = torch.stack([s[t].abs().max().float() for t in ("x", "w", "dy")])
        s["stats"] = torch.zeros(6 * STATS_BYTES, dtype=torch.uint8, device="cuda")
        s["sums"], s["amax"] = _stats_views(s["stats"])
        return s
    s["y"], s["dx"], s["dw"] = _bf16(M, N), _bf16(M, K), _bf16(N, K)
    if kind == "tagged":
        # one workspace for the three calls
        s["ws"] = _bytes(max(api.snip_workspace_size(op, M, N, K, case[t], case[t])[1]
                             for op, t in ((api.OP_FWD, "fwd"), (api.OP_DGRAD, "dgrad"), (api.OP_WGRAD, "wgrad"))))
        return s
    s["stats"] = torch.zeros(6 * STATS_BYTES, dtype=torch.uint8, device="cuda")
    s["sums"], s["amax"] = _stats_views(s["stats"])
    s["ws"] = _bytes(api.snip_linear_fwd_bwd_workspace(M, N, K, case["fwd"], case["dgrad"], case["wgrad"], case["pow2"]))
    return s


# ---- one pass ---------------------------------------------------------------------------------------


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "linear":
        y, dx, dw, _ = api.snip_linear_fwd_bwd(s["x"], s["w"], s["dy"], c["fwd"], c["dgrad"], c["wgrad"], pow2_scale=c["pow2"],
                                               dy_sr_seed=1234567 if c["sr"] else None, y=s["y"], dx=s["dx"], dw=s["dw"],
                                               stats=s["stats"], ws=s["ws"])
        return {"y": y, "dx": dx, "dw": dw, "sums": s["sums"], "amax": s["amax"]}
    if kind == "tagged":
        y, a, b = api.snip_linear_fwd(s["x"], s["w"], c["fwd"], c["fwd"], out=s["y"], ws=s["ws"], want_stats=True)
        dx, d, e = api.snip_linear_dgrad(s["dy"], s["w"], c["dgrad"], c["dgrad"], out=s["dx"], ws=s["ws"], want_stats=True)
        dw, f, g = api.snip_linear_wgrad(s["dy"], s["x"], c["wgrad"], c["wgrad"], out=s["dw"], ws=s["ws"], want_stats=True)
        return {"y": y, "dx": dx, "dw": dw, "stats": [_stats_views(t) for t in (a, b, d, e, f, g)]}
    if kind == "nvfp4":
        y, dx, dw, _ = api.snip_linear_fwd_bwd_nvfp4(s["x"], s["w"], s["dy"], s["bounds"], dy_sr_seed=1234567 if c["sr"] else None,
                                                     stats=s["stats"])
        return {"y": y, "dx": dx, "dw": dw, "sums": s["sums"], "amax": s["amax"]}
    if kind == "forward":
        api.snip_quantize(s["x"], c["fmt"], api.BLOCK_ROW, api.Q_STATS, codes=s["codes"], scales=s["scales"], stats=s["stats"], ws=s["qws"])
        y = api.snip_gemm_quantized(api.OP_FWD, s["x_op"], s["w_op"], (c["M"], c["N"]), out=s["y"], ws=s["gws"])
        return {"y": y, "codes": s["codes"], "scales": s["scales"], "sums": s["sums"], "amax": s["amax"]}
    if kind == "stats":
        return api.snip_layer_stats(X=s["x"], W=s["w"], Y=s["y"], dY=s["dy"], dX=s["dx"], dW=s["dw"], M=c["M"], N=c["N"], K=c["K"],
                                    out=s["out"], ws=s["ws"])
    return api.snip_adamw_sensitivity(s["m"], s["v"], s["g"], 0.9, 0.95, 1e-8, out=s["out"])


def work(case):
    N, K = case["N"], case["K"]
    if case["kind"] == "adamw":
        return {"bytes": (12 if case["grad32"] else 10) * N * K, "flops": 0}
    M = case["M"]
    tensors = 2 * (M * K + N * K + M * N)          # X, W and dY (or Y), bf16
    if case["kind"] == "forward":
        code = 1.0 if case["fmt"] == FP8 else 0.5  # bytes per element of the quantized X and W
        return {"bytes": 2 * M * K + code * (M * K + N * K) + 4 * M * K / 128 + 2 * M * N, "flops": 2 * M * N * K}
    if case["kind"] == "stats":
        return {"bytes": 2 * tensors, "flops": 0}
    return {"bytes": 2 * tensors, "flops": 6 * M * N * K}   # three tensors in, three out, three GEMMs


def tolerance(case):
    if case["kind"] in ("stats", "adamw"):
        return {"rel": 1e-5, "max": 1e-4}     # sums of binary32 terms
    return {"rel": 4e-3, "max": 2e-2}         # bf16 outputs of binary32 sums; codes are whole numbers and stay the same
