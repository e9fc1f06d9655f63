"""Reductions at the edges of their grids: the statistics of a tensor that keeps BF16, the AdamW
sensitivity norm, the layer statistics on the smallest shapes and with norm-only tensors alone."""
import numpy as np
import pytest
import torch

from oracle import snip_oracle as orc
from paper_2602_01410_b200 import workloads as wl
from test_gpu_adamw import moments

pytestmark = pytest.mark.gpu
from gpu_util import to_dev  # noqa: E402

GRID = 6 * 148   # CTAs of a full grid of the AdamW norm


@pytest.fixture(scope="module")
def api():
    from paper_2602_01410_b200 import api as _api
    return _api


# (rows, cols, row stride): one tile, many tiles in one column / row of tiles, ragged tiles; with gaps between the rows
@pytest.mark.parametrize("rows,cols,ld", [(64, 64, 64), (128 * (GRID - 1), 128, 128), (37 * 128, 24 * 128, 24 * 128), (64, (GRID + 1) * 128, (GRID + 1) * 128),
                                          (64, 64, 72), (192, 320, 448), (37 * 128, 24 * 128, 24 * 128 + 8)])
def test_bf16_norm(api, rows, cols, ld):
    rng = np.random.default_rng(rows + cols + ld)
    bits = wl.make_dy(rng, rows, ld)
    x = to_dev(bits)[:, :cols]
    stats = api.snip_quantize(x, 0, 2, api.Q_STATS)[2]
    st = api.stats_to_host(stats)
    v = orc.bf16_to_float(bits[:, :cols])
    assert st["sumsq_x"] == pytest.approx(float(np.square(v.astype(np.float64)).sum()), rel=1e-6)
    assert st["sumsq_err"] == 0.0 and st["amax"] == float(np.abs(v).max())


# four elements per thread and load, two loads per thread: around one CTA, around a full grid's single and double load
@pytest.mark.parametrize("n", [4 * 255, 4 * 257, 4 * 256 * GRID - 4, 4 * 256 * GRID + 4, 4 * 512 * GRID, 4 * 512 * GRID + 4, 4 * 768 * GRID + 1028])
@pytest.mark.parametrize("g_bf16", [False, True])
def test_adamw_norm_around_the_grid(api, n, g_bf16):
    rng = np.random.default_rng(n)
    b1, b2, eps = float(np.float32(0.9)), float(np.float32(0.95)), float(np.float32(1e-8))
    m, v, g = moments(rng, n, steps=2)
    gt = torch.from_numpy(g).cuda()
    if g_bf16:
        gt = gt.to(torch.bfloat16)
        g = gt.float().cpu().numpy()
    out = api.snip_adamw_sensitivity(torch.from_numpy(m).cuda(), torch.from_numpy(v).cuda(), gt, b1, b2, eps)
    assert float(out.cpu()[0]) == pytest.approx(orc.adamw_sensitivity_sumsq(m, v, g, b1, b2, eps), rel=1e-4)


@pytest.mark.parametrize("shape", [(64, 64, 64), (64, 2112, 64), (4160, 192, 320)])
@pytest.mark.parametrize("which", ["all", "norms", "errors", "dY"])
def test_layer_stats_subsets(api, shape, which):
    M, K, N = shape
    rng = np.random.default_rng(M + K + N)
    full = {"X": wl.make_x(rng, M, K), "W": wl.make_w(rng, N, K), "Y": wl.make_x(rng, M, N), "dY": wl.make_dy(rng, M, N),
            "dX": wl.make_dy(rng, M, K), "dW": wl.make_dy(rng, N, K)}
    names = {"all": list(full), "norms": ["Y", "dX", "dW"], "errors": ["X", "W", "dY"], "dY": ["dY"]}[which]
    out = api.snip_layer_stats(**{k: to_dev(full[k]) for k in names}, M=M, N=N, K=K).cpu().numpy()
    for i, name in enumerate(full):
        want = float(np.square(orc.bf16_to_float(full[name]).astype(np.float64)).sum()) if name in names else 0.0
        assert out[i] == pytest.approx(want, rel=1e-4), name
    err = out[6:].reshape(3, 2, 3)
    for t, (name, blocks) in enumerate((("X", (0, 1)), ("W", (2,)), ("dY", (0, 1)))):
        for fmt in (1, 2):
            for b in range(3):
                want = orc.quantize(full[name], fmt, b).sumsq_err if name in names and b in blocks else 0.0
                assert err[t, fmt - 1, b] == pytest.approx(want, rel=1e-4), (name, fmt, b)
