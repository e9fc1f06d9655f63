"""Linear-layer calls as chains of dependent launches: what a caller relies on when the calls follow one another.

Back to back on one workspace, with inputs that the kernel directly ahead has just written, a call gives bit for bit what it
gives alone; so does a replayed graph whose inputs have been replaced in between (a chain member that read an earlier call's
codes, scale factors, bounds or inputs would differ)."""
import numpy as np
import pytest
import torch

from paper_2602_01410_b200 import workloads as wl

pytestmark = pytest.mark.gpu
from gpu_util import to_dev  # noqa: E402

BF16, FP8, FP4 = 0, 1, 2


@pytest.fixture(scope="module")
def api():
    from paper_2602_01410_b200 import api as _api
    return _api


def inputs(M, K, N, seed, factor):
    rng = np.random.default_rng(seed)
    x, w, dy = (to_dev(t) * factor for t in (wl.make_x(rng, M, K, 0.01, 20.0), wl.make_w(rng, N, K), wl.make_dy(rng, M, N)))
    return [x, w, dy, torch.stack([t.abs().max().float() for t in (x, w, dy)])]


def layer(api, kind, M, K, N):
    """(workspace, step): step(tensors, ws) enqueues one layer and returns its outputs, in buffers of their own."""
    if kind == "nvfp4":
        ws = torch.empty(layer_nvfp4_bytes(api, M, K, N), dtype=torch.uint8, device="cuda")
        return ws, lambda t, ws: api.snip_linear_fwd_bwd_nvfp4(t[0], t[1], t[2], t[3], dy_sr_seed=3, ws=ws)
    if kind in ("separate", "tagged"):
        f = (FP8, FP4, FP8) if kind == "separate" else (BF16, BF16, BF16)
        ops = (api.OP_FWD, api.OP_DGRAD, api.OP_WGRAD)
        ws = torch.empty(max(api.snip_workspace_size(op, M, N, K, g, g)[1] for op, g in zip(ops, f)), dtype=torch.uint8, device="cuda")

        def step(t, ws):
            x, w, dy, _ = t
            return (*api.snip_linear_fwd(x, w, f[0], f[0], ws=ws, want_stats=True), *api.snip_linear_dgrad(dy, w, f[1], f[1], ws=ws, want_stats=True),
                    *api.snip_linear_wgrad(dy, x, f[2], f[2], ws=ws, want_stats=True))
        return ws, step
    f, pow2 = {"fp8": ((FP8, FP8, FP8), 0), "fp4": ((FP4, FP4, FP4), 0), "mixed": ((FP8, FP4, FP8), 0), "pow2": ((FP8, FP4, FP4), 1),
               "pow2-32": ((FP4, FP8, FP8), 2)}[kind]
    ws = torch.empty(api.snip_linear_fwd_bwd_workspace(M, N, K, *f, pow2), dtype=torch.uint8, device="cuda")
    return ws, lambda t, ws: api.snip_linear_fwd_bwd(t[0], t[1], t[2], *f, pow2_scale=pow2, dy_sr_seed=3, ws=ws)


def layer_nvfp4_bytes(api, M, K, N):
    import ctypes
    n = ctypes.c_size_t()
    assert api._lib.snip_linear_fwd_bwd_nvfp4_workspace(M, N, K, ctypes.byref(n)) == api.OK
    return n.value


# the quantizers in one launch / in three; the weight gradient sliced (8192 tokens, small weight)
SHAPES = [(512, 384, 640), (1600, 1024, 1216), (8192, 256, 320)]
KINDS = ["fp8", "fp4", "mixed", "pow2", "pow2-32", "nvfp4", "separate", "tagged"]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", KINDS)
def test_calls_back_to_back_on_one_workspace(api, kind, shape):
    sets = [inputs(*shape, 31, 1.0), inputs(*shape, 32, 0.3)]
    want = []
    for s in sets:
        ws, step = layer(api, kind, *shape)
        want.append(step(s, ws))
        torch.cuda.synchronize()
        assert api.snip_poll_status(ws) == api.OK
    ws, step = layer(api, kind, *shape)
    ws.fill_(0xFF)
    now = [torch.empty_like(t) for t in sets[0]]   # every call's inputs in the same place, written just ahead of it
    got = []
    torch.cuda.synchronize()
    for i in range(8):
        for dst, src in zip(now, sets[i % 2]):
            dst.copy_(src)
        got.append(step(now, ws))
    torch.cuda.synchronize()
    assert api.snip_poll_status(ws) == api.OK
    for i, out in enumerate(got):
        for j, (g, ref) in enumerate(zip(out, want[i % 2])):
            assert torch.equal(g.view(torch.uint8), ref.view(torch.uint8)), (i, j)


@pytest.mark.parametrize("shape", SHAPES[:2])
@pytest.mark.parametrize("kind", KINDS)
def test_graph_replays_follow_replaced_inputs(api, kind, shape):
    sets = [inputs(*shape, 41, 1.0), inputs(*shape, 42, 0.3)]
    ws, step = layer(api, kind, *shape)
    want = [step(s, ws) for s in sets]
    now = [t.clone() for t in sets[0]]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            out = step(now, ws)
    got = []
    for i in range(6):   # no synchronisation in between
        for dst, src in zip(now, sets[i % 2]):
            dst.copy_(src)
        graph.replay()
        got.append([t.clone() for t in out])
    torch.cuda.synchronize()
    assert api.snip_poll_status(ws) == api.OK
    for i, o in enumerate(got):
        for j, (g, ref) in enumerate(zip(o, want[i % 2])):
            assert torch.equal(g.view(torch.uint8), ref.view(torch.uint8)), (i, j)


@pytest.mark.parametrize("kind", ["fp8", "pow2", "nvfp4", "separate", "tagged"])
def test_a_refused_call_enqueues_nothing(api, kind):
    # a misaligned output: the call returns an error and leaves workspace and statistics as they were
    M, K, N = 256, 384, 192
    x, w, dy, bounds = inputs(M, K, N, 51, 1.0)
    ws, _ = layer(api, kind, M, K, N)
    ws.fill_(0xA5)
    stats = torch.full((6 * 24 + 16,), 0x5A, dtype=torch.uint8, device="cuda")
    before = ws.clone(), stats.clone()
    off = torch.empty(M * K + M * N + 64, dtype=torch.bfloat16, device="cuda")[4:]   # 8 bytes off
    y, dx, dw = (torch.empty(s, dtype=torch.bfloat16, device="cuda") for s in ((M, N), (M, K), (N, K)))
    p = lambda t: t.data_ptr()
    stream = torch.cuda.current_stream().cuda_stream
    for bad in range(3):
        o = [p(off) if i == bad else p(t) for i, t in enumerate((y, dx, dw))]
        if kind == "nvfp4":
            rc = api._lib.snip_linear_fwd_bwd_nvfp4(p(x), p(w), p(dy), *o, M, N, K, api.OUT_BF16, p(bounds), 0, 0, p(stats), p(ws), ws.numel(), stream)
        elif kind in ("fp8", "pow2"):
            f = (FP8, FP8, FP8) if kind == "fp8" else (FP8, FP4, FP4)
            rc = api._lib.snip_linear_fwd_bwd(p(x), p(w), p(dy), *o, M, N, K, *f, api.OUT_BF16, int(kind == "pow2"), 0, 0, p(stats), p(ws), ws.numel(), stream)
        else:
            f = (FP8, FP4, FP8)[bad] if kind == "separate" else BF16
            fn = (api._lib.snip_linear_fwd, api._lib.snip_linear_dgrad, api._lib.snip_linear_wgrad)[bad]
            a, b = ((x, w), (dy, w), (dy, x))[bad]
            acc = (0,) if bad == 2 else ()
            rc = fn(p(a), p(b), o[bad], M, N, K, f, f, api.OUT_BF16, *acc, p(stats), p(stats) + 32, p(ws), ws.numel(), stream)
        assert rc == api.ERR_ALIGN, bad
    torch.cuda.synchronize()
    assert torch.equal(ws, before[0]) and torch.equal(stats, before[1])
