"""Run by tests/test_bounds_debug_f32tc_gpu.py in a child process with
KSELECT_DEBUG_BOUNDS=1: the FP32 products on the tensor cores in the bounds-checking
build, every tile width, whole and with K divided, every transpose, ragged sizes, rows of
every alignment, a shared operand, values that are computed again, a handle call whose
plan divides K, and a convolution that reads the image.  No access may fall outside the
operands and every result must match the FP64 oracle; then each operand's extent is
declared short, and accesses must be flagged.  Prints one JSON line."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import numpy as np  # noqa: E402
import torch  # noqa: E402

from oracle import gemm as og  # noqa: E402
from oracle import vgg as ov  # noqa: E402
from paper_2008_13145_gb300 import kselect as ks  # noqa: E402
from paper_2008_13145_gb300 import vgg  # noqa: E402
from paper_2008_13145_gb300 import workloads as wl  # noqa: E402
from tests.bounds_debug_check import errors  # noqa: E402

DEPLOY = os.path.join(os.path.dirname(os.path.abspath(vgg.__file__)), "deploy", "f32.json")


def run(bn, splits, sh, pad, beta, lost, shared=False, seed=0):
    A, B, C0 = wl.gemm_inputs(sh, seed=seed, beta_nonzero=beta != 0, ld_multiple=pad)
    if lost:
        A[0, -1, 0] = B[-1, -1, 0] = np.float32(1.2345e-36)
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.from_numpy(np.nan_to_num(C0, nan=0.0)).cuda()
    ks.f32tc_selftest(bn, splits, sh.transA, sh.transB, sh.M, sh.N, sh.K, -0.5, tA, A.shape[2],
                      0 if shared else A.shape[1] * A.shape[2], tB, B.shape[2], B.shape[1] * B.shape[2], beta, C,
                      C0.shape[2], C0.shape[1] * C0.shape[2], sh.batch)
    torch.cuda.synchronize()
    if shared:
        A = np.repeat(A[:1], sh.batch, axis=0)
    ref, den = og.gemm(sh.transA, sh.transB, sh.M, sh.N, sh.K, -0.5, A, B, beta, C0 if beta else None)
    return og.error_ratio(C.cpu().numpy()[:, :, :sh.N], ref, den)


def handle_calls():
    """(errors relative to the FP64 results, K ranges of the plan) of a split product and of a convolution."""
    h = ks.Handle(json.load(open(DEPLOY)))
    M, N, K = 512, 384, 4096
    _, splits = ks.f32tc_choice(ks.select_kernel(h, M, N, K), M, N, K)
    rng = np.random.default_rng(1)
    A, B = (rng.uniform(-1, 1, s).astype(np.float32) for s in ((1, M, K), (1, K, N)))
    C = torch.zeros((1, M, N), device="cuda")
    ks.gemm(h, "N", "N", M, N, K, 1.0, torch.from_numpy(A).cuda(), K, torch.from_numpy(B).cuda(), N, 0.0, C, N)
    ref, den = og.gemm("N", "N", M, N, K, 1.0, A, B, nthreads=og.max_threads())
    worst = og.error_ratio(C.cpu().numpy(), ref, den)
    n, H, W, ch, co = 2, 70, 75, 128, 264
    x = np.abs(rng.standard_normal((n, H, W, ch))).astype(np.float32)
    w = rng.standard_normal((co, 9 * ch)).astype(np.float32)
    x[0, 5, 6, 7] = np.float32(1.2345e-36)
    tx, tw = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
    col = torch.full((n * H * W, 9 * ch), float("nan"), device="cuda")
    out = torch.empty((n * H * W, co), device="cuda")
    ks.conv3x3(h, tx, n, H, W, ch, tw, co, None, False, col, 9 * ch, out)
    assert bool(torch.isnan(col).all()), "the convolution wrote its neighbourhoods out"
    rows = ov.im2col3x3(x.astype(np.float64))
    ref, den = rows @ w.astype(np.float64).T, np.abs(rows) @ np.abs(w.astype(np.float64)).T
    return max(worst, float(np.max(np.abs(out.cpu().numpy() - ref) / den))), splits


def main():
    errors(clear=True)
    worst, cases = 0.0, 0
    for bn in (64, 128, 256):
        for i, (M, N, K, batch, pad) in enumerate([(37, 45, 29, 2, 1), (300, 261, 97, 2, 4), (140, 520, 200, 1, 8)]):
            for t in ("NN", "NT", "TN", "TT"):
                for splits in (1, 3):
                    for lost in (False, True):
                        sh = wl.Shape(M, N, K, batch, t[0], t[1])
                        worst = max(worst, run(bn, splits, sh, pad, 0.25 * (i % 2), lost, shared=i == 1, seed=i))
                        cases += 1
    err, splits = handle_calls()
    found = errors(clear=True)
    flagged = []
    for op in range(3):  # the checker itself: one operand's extent declared 16 bytes short
        for lost in (False, True):
            ks.check(ks._lib.kselect_debug_shrink_extents(*(16 * (op == o) for o in range(3))), "shrink")
            run(128, 1, wl.Shape(64, 64, 64, 1, "N", "N"), 4, 0.0, lost)
            flagged.append(errors(clear=True))
    ks.check(ks._lib.kselect_debug_shrink_extents(0, 0, 0), "kselect_debug_shrink_extents")
    print(json.dumps({"cases": cases, "handle_splits": splits, "out_of_bounds": found,
                      "worst_error_ratio": max(worst, err), "flagged": flagged}))


if __name__ == "__main__":
    main()
