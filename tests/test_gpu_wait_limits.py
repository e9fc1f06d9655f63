"""Waits that run out in every GEMM form and inside chains of launches (test_gpu_gemm_kernels.py has the stand-alone forward product on
one CTA and on a pair).

The condition is made on the host: each stage's barrier expects 16 bytes more than its copies deliver, so every copy lands but the
phase never completes.  With the wait limit at 20 ms each kernel gives up by itself, releases its tensor memory and raises the status
word; nothing traps, faults or spins without a bound.  Afterwards the same call on the same workspace gives what it gave before."""
import pytest
import torch

pytestmark = pytest.mark.gpu
from test_gpu_chain import BF16, FP4, FP8, api, inputs, layer  # noqa: E402,F401


@pytest.fixture
def hooks(api):  # noqa: F811
    def run_out(on):
        api.snip_debug_set(api.DEBUG_WAIT_LIMIT_NS, 20_000_000 if on else 2_000_000_000)
        api.snip_debug_set(api.DEBUG_TX_SKEW_BYTES, 16 if on else 0)

    yield run_out
    run_out(False)
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_AUTO)


def check(api, hooks, ws, call):  # noqa: F811
    def once():
        out = call()
        torch.cuda.synchronize()
        return [t.clone() for t in out if t is not None]

    want = once()
    assert api.snip_poll_status(ws) == api.OK
    hooks(True)
    during = once()
    hooks(False)
    assert api.snip_poll_status(ws) == api.ERR_TIMEOUT
    got = once()
    assert api.snip_poll_status(ws) == api.OK
    for g, ref in zip(got, want):
        assert torch.equal(g.view(torch.uint8), ref.view(torch.uint8))
    return want, during


# paper-rule products: 1 = one CTA, 2 = pair, 3 = 128-wide tiles; power-of-two and two-level products choose by shape (9 x 9 tiles of
# 256 x 256: pairs, in all three products)
@pytest.mark.parametrize("kind,choice,shape", [(k, c, (512, 384, 256)) for k in ("fp8", "fp4", "mixed") for c in (1, 2, 3)] +
                         [(k, 0, s) for k in ("pow2", "pow2-32", "nvfp4") for s in ((512, 384, 256), (2304, 2304, 2304))] +
                         [(k, c, (8192, 256, 320)) for k in ("fp8", "fp4") for c in (0, 1)])   # the weight gradient sliced: in clusters, through the workspace
def test_chained_layer(api, hooks, kind, choice, shape):  # noqa: F811
    t = inputs(*shape, 61, 1.0)
    ws, step = layer(api, kind, *shape)
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, choice)
    want, during = check(api, hooks, ws, lambda: step(t, ws))
    if shape[0] == 8192:
        assert api.snip_debug_last_gemm()[2:] == ((4, 4) if choice == 0 else (4, 1))
    # the quantizers and their statistics are not held up
    assert torch.equal(during[3], want[3])


# one CTA per tile; pairs (10 x 8 tiles of 256 x 256); slices of the contraction (8192 long) in the weight gradient
@pytest.mark.parametrize("want_stats", [False, True])
@pytest.mark.parametrize("op,shape", [(0, (256, 192, 320)), (1, (256, 192, 320)), (2, (256, 192, 320)), (0, (2560, 128, 2048)), (1, (2560, 2048, 128)),
                                      (2, (128, 2048, 2560)), (2, (8192, 256, 256))])
def test_bf16_products(api, hooks, op, shape, want_stats):  # noqa: F811
    M, K, N = shape
    x, w, dy, _ = inputs(M, K, N, 62, 1.0)
    fn, a, b = ((api.snip_linear_fwd, x, w), (api.snip_linear_dgrad, dy, w), (api.snip_linear_wgrad, dy, x))[op]
    ws = torch.full((api.snip_workspace_size(op, M, N, K, BF16, BF16)[1],), 0xFF, dtype=torch.uint8, device="cuda")
    check(api, hooks, ws, lambda: fn(a, b, BF16, BF16, ws=ws, want_stats=want_stats))


@pytest.mark.parametrize("op", [0, 1, 2])
@pytest.mark.parametrize("fmt", [FP8, FP4])
@pytest.mark.parametrize("choice", [1, 2, 3])
def test_separate_products(api, hooks, choice, fmt, op):  # noqa: F811
    M, K, N = 512, 384, 256
    x, w, dy, _ = inputs(M, K, N, 63, 1.0)
    fn, a, b = ((api.snip_linear_fwd, x, w), (api.snip_linear_dgrad, dy, w), (api.snip_linear_wgrad, dy, x))[op]
    ws = torch.full((api.snip_workspace_size(op, M, N, K, fmt, fmt)[1],), 0xFF, dtype=torch.uint8, device="cuda")
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, choice)
    check(api, hooks, ws, lambda: fn(a, b, fmt, fmt, ws=ws))


def test_narrow_product_of_quantized_operands(api, hooks):  # noqa: F811
    M, K, N = 512, 384, 256   # a call of its own: the kernel clears the status word itself
    x, w, _, _ = inputs(M, K, N, 64, 1.0)
    cx, sx, _, _ = api.snip_quantize(x, FP8, api.BLOCK_ROW)
    cw, sw, _, _ = api.snip_quantize(w, FP8, api.BLOCK_BLK)
    a, b = api.make_qtensor(cx, sx, M, K, FP8, api.BLOCK_ROW), api.make_qtensor(cw, sw, N, K, FP8, api.BLOCK_BLK)
    ws = torch.full((256,), 0xFF, dtype=torch.uint8, device="cuda")
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_NARROW)
    check(api, hooks, ws, lambda: [api.snip_gemm_quantized(api.OP_FWD, a, b, (M, N), api.OUT_FP32, ws=ws)])


# A tile of the weight gradient whose slices are the CTAs of a cluster (128-wide tiles; 8192 tokens: four slices, 3072: three): the hook holds
# up the first slice alone.  The others have their sums, but none of a cluster may store its share of a tile that one slice is missing from;
# above all nothing may be added to a caller's gradient.
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("fmt", [FP8, FP4])
@pytest.mark.parametrize("M", [3072, 8192])
def test_slices_of_a_tile_that_one_slice_is_missing_from(api, hooks, M, fmt, accumulate):  # noqa: F811
    K, N = 320, 256
    x, _, dy, _ = inputs(M, K, N, 65, 1.0)
    (cd, sd, _, _), (cx, sx, _, _) = (api.snip_quantize(t, fmt, api.BLOCK_COL, api.Q_TRANSPOSED) for t in (dy, x))
    a, b = api.make_qtensor(cd, sd, M, N, fmt, api.BLOCK_COL, True), api.make_qtensor(cx, sx, M, K, fmt, api.BLOCK_COL, True)
    ws = torch.full((api.snip_workspace_size(api.OP_WGRAD, M, N, K, fmt, fmt)[0],), 0xFF, dtype=torch.uint8, device="cuda")
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_NARROW)
    start = torch.randn(N, K, device="cuda")

    def call():
        return [api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32, accumulate=accumulate, out=start.clone(), ws=ws)]
    _, during = check(api, hooks, ws, call)
    assert torch.equal(during[0], start)
