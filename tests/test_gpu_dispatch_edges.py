"""One layer's forward and both gradients at the sizes where the launch plan changes, against the CPU oracle: the three
quantizers in one launch or in three, the hardware-scaled products on single CTAs or on pairs.

Bar: FP32 output within 1e-5 (relative Frobenius) of the float64 oracle, statistics within 1e-4."""
import numpy as np
import pytest
import torch

from oracle import snip_oracle as orc
from paper_2602_01410_b200 import workloads as wl

pytestmark = pytest.mark.gpu
from gpu_util import rel_fro, to_dev  # noqa: E402

FP8, FP4 = 1, 2
ROW, COL, BLK = 0, 1, 2


@pytest.fixture(scope="module")
def api():
    from paper_2602_01410_b200 import api as _api
    return _api


# 128x128 tiles of X + W + dY around two per SM (296): 12 x 8 + 8 x 9 + 12 x 9 = 276; with ragged edges 13 x 8 + 8 x 9 + 13 x 9 = 293;
# 13 x 8 + 8 x 10 + 13 x 10 = 314
@pytest.mark.parametrize("shape", [(64, 64, 64), (1536, 1024, 1152), (1600, 960, 1088), (1600, 1024, 1216)])
@pytest.mark.parametrize("triple,seed", [((FP8, FP8, FP8), None), ((FP8, FP4, FP8), 5), ((FP4, FP8, FP4), 6), ((FP4, FP4, FP4), 7)])
def test_quantizers_in_one_launch_or_three(api, shape, triple, seed):
    M, K, N = shape
    rng = np.random.default_rng(M + K + N)
    x, w, dy = wl.make_x(rng, M, K, 0.01, 20.0), wl.make_w(rng, N, K), wl.make_dy(rng, M, N)
    ff, fd, fw = triple
    y, dx, dw, st = api.snip_linear_fwd_bwd(to_dev(x), to_dev(w), to_dev(dy), ff, fd, fw, api.OUT_FP32, dy_sr_seed=seed)
    torch.cuda.synchronize()
    sr = lambda fmt: seed if fmt == FP4 else None
    q = (orc.quantize(x, ff, ROW), orc.quantize(x, fw, COL), orc.quantize(w, ff, BLK), orc.quantize(w, fd, BLK),
         orc.quantize(dy, fd, ROW, sr_seed=sr(fd)), orc.quantize(dy, fw, COL, sr_seed=sr(fw)))
    want = (orc.gemm_fwd(q[0].xhat, q[2].xhat), orc.gemm_dgrad(q[4].xhat, q[3].xhat), orc.gemm_wgrad(q[5].xhat, q[1].xhat))
    for name, g, ref in zip(("fwd", "dgrad", "wgrad"), (y, dx, dw), want):
        assert rel_fro(g.cpu().numpy(), ref) <= 1e-5, name
    for i, ref in enumerate(q):
        s = api.stats_to_host(st[24 * i:24 * i + 24])
        assert s["sumsq_x"] == pytest.approx(ref.sumsq_x, rel=1e-4) and s["sumsq_err"] == pytest.approx(ref.sumsq_err, rel=1e-4), i


# outputs of 256x256 tiles around half as many as SMs (37 x 2 = 74), rows ending inside the second half of a tile
@pytest.mark.parametrize("M", [36 * 256, 36 * 256 + 64, 36 * 256 + 192])
@pytest.mark.parametrize("fmt,pow2", [(FP8, 1), (FP4, 1), (FP8, 2), (FP4, 2)])
def test_hardware_scaled_products_in_pairs(api, M, fmt, pow2):
    K, N = 320, 448
    rng = np.random.default_rng(M + fmt)
    x, w, dy = wl.make_x(rng, M, K, 0.01, 20.0), wl.make_w(rng, N, K), wl.make_dy(rng, M, N)
    y, dx, dw, _ = api.snip_linear_fwd_bwd(to_dev(x), to_dev(w), to_dev(dy), fmt, fmt, fmt, api.OUT_FP32, pow2_scale=pow2)
    torch.cuda.synchronize()
    want = (orc.linear_fwd(x, w, fmt, fmt, pow2_scale=pow2)[0], orc.linear_dgrad(dy, w, fmt, fmt, pow2_scale=pow2)[0],
            orc.linear_wgrad(dy, x, fmt, fmt, pow2_scale=pow2)[0])
    for name, g, ref in zip(("fwd", "dgrad", "wgrad"), (y, dx, dw), want):
        assert rel_fro(g.cpu().numpy(), ref) <= 1e-5, name


@pytest.mark.parametrize("M", [36 * 256, 36 * 256 + 64])
def test_two_level_products_in_pairs(api, M):
    K, N = 320, 448
    rng = np.random.default_rng(M)
    x, w, dy = wl.make_x(rng, M, K, 0.01, 20.0), wl.make_w(rng, N, K), wl.make_dy(rng, M, N)
    bounds = torch.tensor([float(np.abs(orc.bf16_to_float(t)).max()) for t in (x, w, dy)], dtype=torch.float32, device="cuda")
    y, dx, dw, _ = api.snip_linear_fwd_bwd_nvfp4(to_dev(x), to_dev(w), to_dev(dy), bounds, api.OUT_FP32)
    torch.cuda.synchronize()
    want = (orc.linear_nvfp4("fwd", x, w)[0], orc.linear_nvfp4("dgrad", dy, w)[0], orc.linear_nvfp4("wgrad", dy, x)[0])
    for name, g, ref in zip(("fwd", "dgrad", "wgrad"), (y, dx, dw), want):
        assert rel_fro(g.cpu().numpy(), ref) <= 1e-5, name
