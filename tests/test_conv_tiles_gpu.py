"""The convolution that reads the image itself at every tile width, whole and with K divided,
against its separate steps in FP64; on values that do not split; and that a handle call
takes it (the im2col scratch stays as it was) where it should."""
import json

import numpy as np
import pytest

from oracle import vgg as ov
from tests.test_f32tc_gpu import DEPLOY

pytestmark = pytest.mark.gpu

# Columns one position high or wide, the fewest channels, several images to a tile, tiles
# across image ends, one image in several tiles, outputs that no vector access allows.
CASES = [(1, 300, 1, 32, 64), (1, 1, 300, 32, 70), (7, 5, 6, 32, 130), (2, 19, 15, 64, 257), (1, 40, 33, 32, 61),
         (3, 1, 1, 96, 8)]


def data(n, H, W, C, Cout):
    rng = np.random.default_rng(H * W + C)
    x = np.abs(rng.standard_normal((n, H, W, C))).astype(np.float32)
    w = (rng.standard_normal((Cout, 9 * C)) * np.sqrt(2.0 / (9 * C))).astype(np.float32)
    return x, w, rng.standard_normal(Cout).astype(np.float32)


def run(lib, bn, splits, x, w, b, relu):
    import torch
    n, H, W, C = x.shape
    Cout = w.shape[0]
    out = torch.full((n * H * W + 1, Cout), float("nan"), device="cuda")
    tx, tw = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
    lib.conv3x3_selftest(bn, splits, tx, n, H, W, C, tw, Cout, None if b is None else torch.from_numpy(b).cuda(), relu,
                         out)
    torch.cuda.synchronize()
    assert lib.device_status() == 0
    got = out.cpu().numpy()
    assert np.all(np.isnan(got[-1]))
    return got[:-1]


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("splits", [1, 3])
@pytest.mark.parametrize("lost", [False, True])
def test_against_separate_steps(lib, bn, splits, lost):
    for n, H, W, C, Cout in CASES:
        x, w, b = data(n, H, W, C, Cout)
        if lost:  # low bits below BF16's range: the tiles are computed again
            x[0, H // 2, W // 2, 3] = x[-1, -1, -1, -1] = np.float32(1.2345e-36)
        rows = ov.im2col3x3(x.astype(np.float64))
        ref, den = rows @ w.astype(np.float64).T, np.abs(rows) @ np.abs(w.astype(np.float64)).T
        for bias, relu in ((b, True), (b, False), (None, True), (None, False)):
            want = ref + (0 if bias is None else bias.astype(np.float64))
            want = np.maximum(want, 0) if relu else want
            got = run(lib, bn, splits, x, w, bias, relu)
            # the FP32 products' tolerance of the library, on |A||w| + |bias|
            assert np.all(np.abs(got - want) <= 1e-5 * (den + (0 if bias is None else np.abs(bias)))), (n, H, W, C, Cout)


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("splits", [1, 3])
def test_infinity_and_nan_with_bias_and_relu(lib, bn, splits):
    """As the separate steps give them: im2col, an FMA chain, bias and ReLU (which takes NaN to 0)."""
    import torch
    x, w, b = data(2, 19, 15, 64, 257)
    x[1, 3, 4, 5], x[0, 18, 14, 0], w[3, 70] = np.inf, np.nan, -np.inf
    M, K, Cout = 2 * 19 * 15, 9 * 64, 257
    tx, tw, tb = (torch.from_numpy(v).cuda() for v in (x, w, b))
    col, want = torch.empty((M, K), device="cuda"), torch.empty((M, Cout), device="cuda")
    lib.im2col3x3(tx, 2, 19, 15, 64, col, K)
    lib.gemm_with_config(533, "N", "T", M, Cout, K, 1.0, col, K, tw, K, 0.0, want, Cout)
    for relu in (True, False):
        ref = want.clone()
        lib.bias_act(ref, M, Cout, Cout, tb, relu)
        ref, got = ref.cpu().numpy(), run(lib, bn, splits, x, w, b, relu)
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
        fine = np.isfinite(ref)
        # sums of 576 terms of about 0.05 in either order
        assert np.max(np.abs(got - ref)[fine]) <= 1e-4


def test_refusals(lib):
    import torch
    x, w, out = (torch.zeros(5000, device="cuda") for _ in range(3))
    for args, status in (((64, 1, x, 1, 2, 2, 33, w, 8), -2), ((64, 1, x[1:], 1, 2, 2, 32, w, 8), -2),
                         ((96, 1, x, 1, 2, 2, 32, w, 8), -1), ((64, 17, x, 1, 2, 2, 32, w, 8), -1),
                         ((64, 1, x, 0, 2, 2, 32, w, 8), -1)):
        with pytest.raises(lib.KSelectError) as e:
            lib.conv3x3_selftest(*args, None, False, out)
        assert e.value.status == status


# Every layer shape here reads the image itself: the scratch of the neighbourhoods stays NaN.
@pytest.mark.parametrize("n,H,W,C,Cout", [(2, 70, 75, 128, 264), (1, 14, 14, 512, 512), (16, 112, 112, 64, 128),
                                          (1, 200, 52, 3, 64)])
def test_handle_call_leaves_the_scratch_alone(lib, n, H, W, C, Cout):
    import os
    import torch
    h = lib.Handle(json.load(open(os.path.join(DEPLOY, "f32.json"))))
    x, w = torch.rand((n, H, W, C), device="cuda"), torch.rand((Cout, 9 * C), device="cuda")
    ld = -(-9 * C // 4) * 4
    col = torch.full((n * H * W, ld), float("nan"), device="cuda")
    out = torch.full((n * H * W, Cout), float("nan"), device="cuda")
    lib.conv3x3(h, x, n, H, W, C, w, Cout, None, True, col, ld, out)
    torch.cuda.synchronize()
    assert bool(torch.isnan(col).all()) and not bool(torch.isnan(out).any())
