"""The 3 x 3 convolution that reads the image itself against its three separate steps in
FP64 (im2col, product, bias + ReLU), where a K chunk, a tile or the image ends."""
import json
import os

import numpy as np
import pytest

from oracle import vgg as ov
from paper_2008_13145_gb300 import vgg

pytestmark = pytest.mark.gpu
DEPLOY = os.path.join(os.path.dirname(os.path.abspath(vgg.__file__)), "deploy")


# Images, height, width, channels, outputs: rows of one position, tiles across image ends,
# every tile width (64, 128, 256 x 256), K split, the smallest channel count, sizes that
# stay with the separate steps (little work), and few channels.
@pytest.mark.parametrize("n,H,W,C,Cout", [(1, 9, 1, 32, 700), (3, 37, 41, 64, 64), (2, 61, 50, 96, 130),
                                          (2, 70, 75, 128, 264), (1, 14, 14, 512, 512), (9, 33, 35, 32, 60),
                                          (2, 12, 10, 3, 64), (1, 4, 4, 32, 8),
                                          (1, 200, 52, 3, 64), (3, 61, 60, 1, 16), (2, 80, 64, 4, 256),
                                          (2, 99, 100, 2, 48)])
@pytest.mark.parametrize("deploy", ["f32.json", "f32mix.json"])
def test_against_separate_steps(lib, n, H, W, C, Cout, deploy):
    import torch
    h = lib.Handle(json.load(open(os.path.join(DEPLOY, deploy))))
    rng = np.random.default_rng(C)
    x = np.abs(rng.standard_normal((n, H, W, C))).astype(np.float32)
    w = (rng.standard_normal((Cout, 9 * C)) * np.sqrt(2.0 / (9 * C))).astype(np.float32)
    b = rng.standard_normal(Cout).astype(np.float32)
    tx, tw, tb = (torch.from_numpy(v).cuda() for v in (x, w, b))
    ld = -(-9 * C // 4) * 4
    col = torch.full((n * H * W, ld), float("nan"), device="cuda")
    A = ov.im2col3x3(x.astype(np.float64))
    ref, den = A @ w.astype(np.float64).T, np.abs(A) @ np.abs(w.astype(np.float64)).T
    for bias, relu in ((b, True), (None, False)):
        out = torch.full((n * H * W + 1, Cout), float("nan"), device="cuda")
        lib.conv3x3(h, tx, n, H, W, C, tw, Cout, None if bias is None else tb, relu, col, ld, out)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        want = ref if bias is None else ref + bias.astype(np.float64)
        want = np.maximum(want, 0) if relu else want
        # the FP32 products' tolerance of the library, on |A||w| + |bias|
        assert np.all(np.abs(got[:-1] - want) <= 1e-5 * (den + (0 if bias is None else np.abs(bias))))
        assert np.all(np.isnan(got[-1]))


def test_infinite_pixel_and_weight(lib):
    """An infinite pixel reaches its neighbours only; an infinite weight meets the zero padding as it does in
    the separate steps."""
    import torch
    h = lib.Handle(json.load(open(os.path.join(DEPLOY, "f32.json"))))
    n, H, W, C, Cout = 2, 60, 50, 64, 128
    g = torch.Generator("cuda").manual_seed(0)
    x = torch.rand((n, H, W, C), generator=g, device="cuda")
    w = torch.rand((Cout, 9 * C), generator=g, device="cuda") - 0.5
    x[1, 30, 20, 5] = float("inf")
    w[3, 70] = float("-inf")
    col = torch.empty((n * H * W, 9 * C), device="cuda")
    out, want = torch.empty((2, n * H * W, Cout), device="cuda")
    lib.conv3x3(h, x, n, H, W, C, w, Cout, None, False, col, 9 * C, out)
    lib.im2col3x3(x, n, H, W, C, col, 9 * C)
    lib.gemm_with_config(533, "N", "T", n * H * W, Cout, 9 * C, 1.0, col, 9 * C, w, 9 * C, 0.0, want, Cout)
    torch.cuda.synchronize()
    assert torch.equal(torch.isnan(out), torch.isnan(want)) and torch.equal(torch.isinf(out), torch.isinf(want))
    fine = torch.isfinite(want)
    assert float((out - want)[fine].abs().max()) <= 1e-4
