"""Tile forms of the GEMM kernels at the sizes where their dispatch changes, against the CPU oracle: 128-wide tiles
(forced, and where the library chooses them), the BF16 kernel with operands in either order, and the slices of a last
wave that is just long enough.

Bar: FP32 output within 1e-5 (relative Frobenius) of the float64 oracle, as in test_gpu_gemm.py."""
import numpy as np
import pytest
import torch

from oracle import snip_oracle as orc
from paper_2602_01410_b200 import workloads as wl

pytestmark = pytest.mark.gpu

BF16, FP8, FP4 = 0, 1, 2

from gpu_util import bf16_out_to_f64, rel_fro, to_dev  # noqa: E402


@pytest.fixture(scope="module")
def api():
    from paper_2602_01410_b200 import api as _api
    return _api


def check_three(api, M, K, N, fa, fb, seed):
    rng = np.random.default_rng(seed)
    x, w, dy = wl.make_x(rng, M, K, 0.01, 20.0), wl.make_w(rng, N, K), wl.make_dy(rng, M, N)
    X, W, DY = to_dev(x), to_dev(w), to_dev(dy)
    got = (api.snip_linear_fwd(X, W, fa, fb, api.OUT_FP32)[0], api.snip_linear_dgrad(DY, W, fa, fb, api.OUT_FP32)[0],
           api.snip_linear_wgrad(DY, X, fa, fb, api.OUT_FP32)[0])
    got16 = (api.snip_linear_fwd(X, W, fa, fb, api.OUT_BF16)[0], api.snip_linear_dgrad(DY, W, fa, fb, api.OUT_BF16)[0],
             api.snip_linear_wgrad(DY, X, fa, fb, api.OUT_BF16)[0])
    torch.cuda.synchronize()
    want = (orc.linear_fwd(x, w, fa, fb)[0], orc.linear_dgrad(dy, w, fa, fb)[0], orc.linear_wgrad(dy, x, fa, fb)[0])
    for name, g, h, ref in zip(("fwd", "dgrad", "wgrad"), got, got16, want):
        assert rel_fro(g.cpu().numpy(), ref) <= 1e-5, name
        assert rel_fro(bf16_out_to_f64(h), orc.bf16_to_float(orc.round_to_bf16(ref))) <= 1e-3, name


# (M, K, N): the smallest; ragged rows, columns and contraction around a 128-wide tile; more narrow tiles than SMs;
# a weight gradient in four slices (FP4 x FP4, whose stages are twice as long where the contraction ends in a 64-wide tile: whole)
@pytest.mark.parametrize("fa,fb", [(FP8, FP8), (FP4, FP4), (FP8, FP4), (FP4, FP8)])
@pytest.mark.parametrize("shape", [(64, 64, 64), (192, 320, 448), (1088, 1472, 1984), (4160, 192, 256)])
@pytest.mark.parametrize("choice", ["narrow", "auto"])
def test_narrow_tiles(api, choice, shape, fa, fb):
    api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_NARROW if choice == "narrow" else api.GEMM_KERNEL_AUTO)
    try:
        check_three(api, *shape, fa, fb, 5000 + sum(shape))
    finally:
        api.snip_debug_set(api.DEBUG_GEMM_KERNEL, api.GEMM_KERNEL_AUTO)


# where the library changes between 128- and 256-wide tiles (37 / 38 row tiles x 2 column tiles of 256: half of 148 SMs), and where it
# goes over to CTA pairs (37 x 2 tiles of 256 x 256)
@pytest.mark.parametrize("M", [37 * 128, 38 * 128, 36 * 256 + 64, 37 * 256])
@pytest.mark.parametrize("fmt", [FP8, FP4])
def test_edges_of_the_tile_rule(api, M, fmt):
    check_three(api, M, 192, 512, fmt, fmt, 6000 + M)


# BF16 products read their operands as they lie in memory: every gradient's ragged tiles, a sliced last wave (M = 4160: 65 stages), and
# enough tiles for CTA pairs (37 x 2 of 256 x 256)
@pytest.mark.parametrize("shape", [(64, 64, 64), (192, 320, 448), (4160, 192, 320), (9472, 128, 512), (9408, 512, 192)])
def test_bf16_operand_orders(api, shape):
    check_three(api, *shape, BF16, BF16, 7000 + sum(shape))


def test_bf16_accumulates_into_fp32(api):
    M, K, N = 448, 320, 192
    rng = np.random.default_rng(11)
    x, dy = wl.make_x(rng, M, K, 0.01, 20.0), wl.make_dy(rng, M, N)
    base = torch.randn(N, K, dtype=torch.float32, device="cuda")
    want = base.double().cpu().numpy() + orc.linear_wgrad(dy, x, BF16, BF16)[0]
    out = api.snip_linear_wgrad(to_dev(dy), to_dev(x), BF16, BF16, api.OUT_FP32, accumulate=True, out=base)[0]
    torch.cuda.synchronize()
    assert rel_fro(out.cpu().numpy(), want) <= 1e-5


# FP4 forward, where both widths take the same number of waves or the narrow ones a quarter or a third more: 128 columns; half as many
# again: 192.  (Row tiles of an output of 1536 columns, i.e. 12 narrow or 8 wide tiles each; the counts are for 148 SMs.)
@pytest.mark.parametrize("row_tiles,width", [(22, 128), (58, 128), (42, 128), (132, 128), (32, 192)])
def test_width_of_fp4_tiles_by_waves(api, row_tiles, width):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("wave counts are for 148 SMs")
    M, K, N = 128 * row_tiles, 128, 1536
    X, W = torch.randn(M, K, device="cuda").bfloat16(), torch.randn(N, K, device="cuda").bfloat16()
    api.snip_linear_fwd(X, W, FP4, FP4)
    torch.cuda.synchronize()
    assert api.snip_debug_last_gemm()[0] == width


# ... and the FP4 weight gradient over a token count that ends in a 64-wide tile: 27 x 17 narrow or 27 x 12 wide tiles are four waves or three,
# 192 columns; 20 x 11 or 20 x 8 are two either way, 128 columns.
@pytest.mark.parametrize("rows,cols,width", [(27 * 128, 17 * 128, 192), (20 * 128, 11 * 128, 128)])
def test_width_of_fp4_weight_gradient_tiles_by_waves(api, rows, cols, width):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("wave counts are for 148 SMs")
    DY, X = torch.randn(192, rows, device="cuda").bfloat16(), torch.randn(192, cols, device="cuda").bfloat16()
    api.snip_linear_wgrad(DY, X, FP4, FP4)
    torch.cuda.synchronize()
    assert api.snip_debug_last_gemm()[0] == width
