"""Weight-gradient product with the tiles of its last wave cut into slices of the contraction: the sliced and the
unsliced run against the CPU oracle and against each other, on shapes whose token count (the contraction) is long
enough for two, three and four slices, with ragged row / column / contraction tiles, in every format pair.

Bar: FP32 output within 1e-5 (relative Frobenius) of the float64 oracle, as in test_gpu_gemm.py; sliced runs
repeat bit for bit (the slices are added in slice order, not in order of arrival)."""
import numpy as np
import pytest
import torch

from oracle import snip_oracle as orc
from paper_2602_01410_b200 import workloads as wl

pytestmark = pytest.mark.gpu

FP8, FP4 = 1, 2
PAIRS = [(FP8, FP8), (FP4, FP4), (FP8, FP4), (FP4, FP8)]

from gpu_util import bf16_out_to_f64, rel_fro, to_dev  # noqa: E402


@pytest.fixture(scope="module")
def api():
    from paper_2602_01410_b200 import api as _api
    return _api


@pytest.fixture
def slicing(api):
    def choose(v):
        api.snip_debug_set(api.DEBUG_GEMM_SLICING, v)
    yield choose
    api.snip_debug_set(api.DEBUG_GEMM_SLICING, 1)


def operands(api, M, K, N, fa, fb, seed):
    rng = np.random.default_rng(seed)
    x, dy = wl.make_x(rng, M, K, 0.01, 20.0), wl.make_dy(rng, M, N)
    X, DY = to_dev(x), to_dev(dy)
    cd, sd, _, _ = api.snip_quantize(DY, fa, api.BLOCK_COL, api.Q_TRANSPOSED)
    cx, sx, _, _ = api.snip_quantize(X, fb, api.BLOCK_COL, api.Q_TRANSPOSED)
    a = api.make_qtensor(cd, sd, M, N, fa, api.BLOCK_COL, True)
    b = api.make_qtensor(cx, sx, M, K, fb, api.BLOCK_COL, True)
    return x, dy, a, b, (cd, sd, cx, sx)


# (tokens M, in-features K, out-features N): 4 tiles x 4 slices; 6 ragged tiles x 2 slices (17 stages); 12 tiles with a
# contraction ending in a 64-wide tile; 48 tiles x 3 slices
SHAPES = [(4096, 512, 256), (2176, 448, 320), (3136, 768, 512), (3072, 1536, 1024)]


@pytest.mark.parametrize("fa,fb", PAIRS)
@pytest.mark.parametrize("shape", SHAPES)
def test_sliced_and_unsliced_match_the_oracle(api, slicing, fa, fb, shape):
    M, K, N = shape
    x, dy, a, b, keep = operands(api, M, K, N, fa, fb, 4000 + M + K + N)
    ref = orc.linear_wgrad(dy, x, fa, fb)[0]
    outs = {}
    for mode in (1, 0):
        slicing(mode)
        outs[mode] = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32)
        torch.cuda.synchronize()
        e = rel_fro(outs[mode].cpu().numpy(), ref)
        assert e <= 1e-5, (mode, e)
    # the two differ only in the order of FP32 additions
    assert rel_fro(outs[1].cpu().numpy(), outs[0].cpu().numpy().astype(np.float64)) <= 1e-6
    slicing(1)
    for _ in range(3):
        again = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32)
        torch.cuda.synchronize()
        assert torch.equal(again, outs[1])
    out16 = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_BF16)
    torch.cuda.synchronize()
    assert rel_fro(bf16_out_to_f64(out16), orc.bf16_to_float(orc.round_to_bf16(ref))) <= 1e-3


def test_sliced_accumulate_garbage_workspace_and_minimum_workspace(api, slicing):
    slicing(1)
    M, K, N = 4096, 512, 256
    x, dy, a, b, keep = operands(api, M, K, N, FP8, FP8, 77)
    ref = orc.linear_wgrad(dy, x, FP8, FP8)[0]
    gbytes, _ = api.snip_workspace_size(api.OP_WGRAD, M, N, K, FP8, FP8)
    assert gbytes > (1 << 20)
    # the caller's workspace holds garbage: status word and arrival counters are cleared by the call itself
    ws = torch.full((gbytes,), 0xFF, dtype=torch.uint8, device="cuda")
    out = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32, ws=ws)
    torch.cuda.synchronize()
    assert api.snip_poll_status(ws) == api.OK
    assert rel_fro(out.cpu().numpy(), ref) <= 1e-5
    # accumulate: the slice sums are added to what the output holds
    out2 = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32, accumulate=True, out=out.clone(), ws=ws)
    torch.cuda.synchronize()
    assert rel_fro(out2.cpu().numpy(), 2 * ref) <= 1e-5
    # a 256-byte workspace is still enough (the product then runs unsliced)
    small = torch.full((256,), 0xFF, dtype=torch.uint8, device="cuda")
    out3 = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32, ws=small)
    torch.cuda.synchronize()
    assert api.snip_poll_status(small) == api.OK
    assert rel_fro(out3.cpu().numpy(), ref) <= 1e-5


# Both ways of adding the slices, forced: 128-wide tiles (kernel choice 3) whose slices are the CTAs of a cluster - two, three and four
# of them, ragged tiles on both sides, contractions ending in a 64-wide tile, one group of a tile more for a CTA than for another - and
# 256- / 192-wide tiles (choice 1), which exchange through the workspace.  Partial sums in the workspace are there in the second case only.
@pytest.mark.parametrize("fa,fb", [(FP8, FP8), (FP4, FP4)])
@pytest.mark.parametrize("choice,shape", [(3, (3584, 1024, 1024)), (3, (6208, 704, 448)), (3, (8256, 192, 64)), (3, (8192, 1024, 512)), (3, (4096, 768, 768)), (1, (8192, 448, 320)), (1, (8256, 512, 256))])
def test_cluster_and_workspace_exchange(api, slicing, fa, fb, choice, shape):
    M, K, N = shape
    x, dy, a, b, keep = operands(api, M, K, N, fa, fb, 90 + choice + M + K + N)
    start = torch.randn(N, K, device="cuda")
    ws = torch.full((api.snip_workspace_size(api.OP_WGRAD, M, N, K, fa, fb)[0],), 0xA5, dtype=torch.uint8, device="cuda")
    partials = ws[8448:]   # behind status word and arrival counters
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, choice)
    try:
        outs = {}
        for mode in (0, 1, 1):
            slicing(mode)
            f32 = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32, ws=ws)
            width, _, slices, cluster = api.snip_debug_last_gemm()
            assert (width == 128) == (choice == 3) and cluster == (slices if choice == 3 else 1)
            # (6208 tokens in FP4: 25 stages of 256; 32 clusters of four are close to what the chip holds)
            assert slices in ((1,) if mode == 0 else {(3584, 1024, 1024): (2,), (4096, 768, 768): (3,), (6208, 704, 448): (3 if fa == FP4 else 4,),
                                                      (8192, 1024, 512): (3, 4)}.get(shape, (4,)))
            torch.cuda.synchronize()
            assert bool((partials == 0xA5).all()) == (choice == 3 or not outs)
            acc = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32, accumulate=True, out=start.clone())
            b16 = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_BF16)
            torch.cuda.synchronize()
            assert torch.equal(acc, start + f32) and torch.equal(b16, f32.bfloat16())
            if mode and mode in outs:
                assert torch.equal(f32, outs[1])     # whatever the order of arrival
            outs[mode] = f32.clone()
    finally:
        api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_AUTO)
    # they differ in the order of FP32 additions only: a few units in the last place of sums over at most 65 chunks
    assert not torch.equal(outs[1], outs[0])
    assert rel_fro(outs[1].cpu().numpy(), outs[0].cpu().numpy().astype(np.float64)) <= 1e-6


# Clusters of three in numbers that only an idle device has room for (45 of 45): behind another kernel the last ones wait for a whole
# tile's time.  4096 tokens are enough for four slices; from 34 tiles or so on there are three, and never more of them than nine tenths of
# the SMs hold.
@pytest.mark.parametrize("fmt", [FP8, FP4])
def test_clusters_of_three_leave_room(api, fmt):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M, K = 4096, 128
    seen = set()
    for tiles in range(30, 50):
        x, dy, a, b, keep = operands(api, M, K, 128 * tiles, fmt, fmt, tiles)
        api.snip_gemm_quantized(api.OP_WGRAD, a, b, (128 * tiles, K))
        width, ctas, slices, cluster = api.snip_debug_last_gemm()
        assert (width, ctas) == (128, 1) and cluster == slices
        assert slices != 3 or 3 * tiles <= 0.9 * sms, tiles
        seen.add(slices)
    torch.cuda.synchronize()
    assert seen == {2, 3, 4}


# Clusters, or more slices and the exchange through the workspace, by the length of the contraction: (chunks, tiles) -> (slices, CTAs of a
# cluster), sums against the unsliced product as above.  (For 148 SMs in GPCs that hold more than 32 clusters of four.)
@pytest.mark.parametrize("chunks,tiles,want", [(23, 10, (2, 2)), (22, 10, (1, 1)), (64, 45, (2, 2)), (118, 45, (3, 1)), (118, 42, (3, 1)), (118, 36, (3, 3)), (256, 36, (4, 1)), (256, 30, (4, 4))])
def test_exchange_by_the_length_of_the_contraction(api, slicing, chunks, tiles, want):
    M, K, N = 128 * chunks, 128, 128 * tiles
    x, dy, a, b, keep = operands(api, M, K, N, FP8, FP8, chunks + tiles)
    got = {}
    for mode in (0, 1):
        slicing(mode)
        got[mode] = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32)
    torch.cuda.synchronize()
    assert api.snip_debug_last_gemm() == (128, 1, *want)
    # the order of FP32 additions only, over at most 256 chunks (as in test_cluster_and_workspace_exchange, whose bound is for 65)
    assert rel_fro(got[1].cpu().numpy(), got[0].cpu().numpy().astype(np.float64)) <= 2e-6


# In a layer the product starts beside the input gradient: (tokens, in, out), FP8 -> slices.  Whole tiles where they fit on the SMs that are
# free then and slices do not; slices where neither fits, both fit, or the contraction is long.  (Counts are for 148 SMs.)
@pytest.mark.parametrize("shape,slices", [((3072, 256, 4608), 1), ((3072, 1024, 1024), 1), ((3072, 4608, 256), 1), ((3584, 1152, 1024), 2),
                                          ((3072, 512, 512), 3), ((5120, 256, 4608), 2)])
def test_slices_of_a_product_that_starts_beside_others(api, shape, slices):
    M, K, N = shape
    rng = np.random.default_rng(sum(shape))
    x, w, dy = to_dev(wl.make_x(rng, M, K, 0.01, 20.0)), to_dev(wl.make_w(rng, N, K)), to_dev(wl.make_dy(rng, M, N))
    _, _, dw, _ = api.snip_linear_fwd_bwd(x, w, dy, FP8, FP8, FP8, api.OUT_FP32)
    assert api.snip_debug_last_gemm()[:3] == (128, 1, slices)
    api.snip_linear_wgrad(dy, x, FP8, FP8)
    assert api.snip_debug_last_gemm()[2] > 1     # on its own it is sliced
    api.snip_debug_set(api.DEBUG_GEMM_SLICING, 0)
    try:
        ref = api.snip_linear_wgrad(dy, x, FP8, FP8, api.OUT_FP32)[0]
        torch.cuda.synchronize()
    finally:
        api.snip_debug_set(api.DEBUG_GEMM_SLICING, 1)
    # the order of FP32 additions over at most 40 chunks (as above)
    assert rel_fro(dw.cpu().numpy(), ref.cpu().numpy().astype(np.float64)) <= 1e-6


# 128-wide tiles that exchange through the workspace: more of them than SMs, so that only the last wave's are sliced (160 tiles: 148 and twelve,
# these in three and four slices; ragged: 148 and twenty; a contraction that ends in a 64-wide tile, in FP4 stages of 256).
@pytest.mark.parametrize("fa,fb", [(FP8, FP8), (FP4, FP4)])
@pytest.mark.parametrize("shape,slices", [((3840, 640, 4096), 3), ((4096, 640, 4096), 4), ((4096, 704, 3520), 4), ((8256, 640, 4096), 4)])
def test_last_wave_of_narrow_tiles(api, slicing, fa, fb, shape, slices):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("wave counts are for 148 SMs")
    M, K, N = shape
    x, dy, a, b, keep = operands(api, M, K, N, fa, fb, 600 + M + K + N)
    ref = orc.linear_wgrad(dy, x, fa, fb)[0]
    start = torch.randn(N, K, device="cuda")
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_NARROW)
    try:
        out = [api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32) for _ in range(3)]
        plan = api.snip_debug_last_gemm()
        acc = api.snip_gemm_quantized(api.OP_WGRAD, a, b, (N, K), api.OUT_FP32, accumulate=True, out=start.clone())
        torch.cuda.synchronize()
    finally:
        api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_AUTO)
    assert plan == (128, 1, slices, 1)
    assert rel_fro(out[0].cpu().numpy(), ref) <= 1e-5
    assert torch.equal(out[1], out[0]) and torch.equal(out[2], out[0]) and torch.equal(acc, start + out[0])
