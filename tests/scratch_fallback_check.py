"""Run by tests/test_scratch_fallback_gpu.py in a child process with KSELECT_DEBUG_BOUNDS=1:
handle calls whose tensor-core plan divides K while the scratch allocation fails.  Prints
one JSON line."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import torch  # noqa: E402

from paper_2008_13145_gb300 import kselect as ks  # noqa: E402


def fail(n):
    ks.check(ks._lib.kselect_debug_fail_scratch(n), "kselect_debug_fail_scratch")


def error(C, A, B):
    ref = A.double() @ B.double()
    return float(((C.double() - ref).abs() / (A.double().abs() @ B.double().abs())).max())


def main():
    M, N, K = 512, 384, 4096
    A, B = torch.rand((M, K), device="cuda") - 0.5, torch.rand((K, N), device="cuda") - 0.5
    C = torch.full((M, N), float("nan"), device="cuda")
    h = ks.Handle({"precision": ks.PREC_F32, "config_ids": [525]})  # whole K: needs no scratch
    out = {"plan_splits": ks.f32tc_choice(525, M, N, K)[1]}
    want = C.clone()
    ks.gemm_with_config(525, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, want, N)
    fail(1)
    ks.gemm(h, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C, N)
    out["gemm_same_as_config"] = torch.equal(C, want)
    ks.gemm(h, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C, N)  # with scratch again
    out["then_tensor_cores"] = not torch.equal(C, want)
    out["errors"] = [error(want, A, B), error(C, A, B)]

    n, H, W, ch, co = 1, 14, 14, 512, 512
    x, w, b = torch.rand((n, H, W, ch), device="cuda"), torch.rand((co, 9 * ch), device="cuda") - 0.5, torch.rand(co, device="cuda")
    rows, ld = n * H * W, 9 * ch
    out["conv_splits"] = ks.f32tc_choice(525, rows, co, ld)[1]
    got = []
    for failures in (0, 2):  # the second: refused to the image form, then to the product of the three steps
        col = torch.full((rows, ld), float("nan"), device="cuda")
        y = torch.full((rows, co), float("nan"), device="cuda")
        fail(failures)
        ks.conv3x3(h, x, n, H, W, ch, w, co, b, True, col, ld, y)
        got.append((y, bool(torch.isnan(col).any())))
    fail(0)
    rel = float((got[0][0] - got[1][0]).abs().max() / got[0][0].abs().max())
    out["conv"] = [got[0][1], got[1][1], rel]

    hs = ks.Handle({"precision": ks.PREC_F32, "config_ids": [2525]})  # the choice divides K itself: refused as ever
    fail(2)
    try:
        ks.gemm(hs, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C, N)
        out["split_choice"] = 0
    except ks.KSelectError as e:
        out["split_choice"] = e.status
    fail(0)
    torch.cuda.synchronize()
    print(json.dumps(out))


if __name__ == "__main__":
    main()
