"""FP32 products on the tensor cores (three-part BF16 splits, K chunks of 32 summed
in FP32) against the FP64 oracle and the SIMT kernels.

Tolerance, relative to |alpha||A||B| + |beta||C0|: the three products left out are
below 2^-24 + 2^-24 + 2^-32 of |xy|; a chunk's accumulator is truncated twice at
the chunk's magnitude (2^-23 each) and ten times at 2^-8 of it; the chunk sums, the
split partials, alpha and beta are each rounded once: (10 + chunks + splits) 2^-24.
"""
import json
import os

import numpy as np
import pytest

from oracle import gemm as og
from paper_2008_13145_gb300 import workloads as wl
from tests.gpu_helpers import Out

pytestmark = pytest.mark.gpu
DEPLOY = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_13145_gb300", "deploy")


@pytest.fixture(scope="module")
def torch():
    import torch as t
    return t


def tolerance(K, splits):
    return (10 + -(-K // 32) + splits) * 2.0 ** -24


def run(lib, torch, bn, splits, sh, A, B, C0, alpha, beta):
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    out = Out(torch, C0, beta, sh.N)
    lib.f32tc_selftest(bn, splits, sh.transA, sh.transB, sh.M, sh.N, sh.K, alpha, tA, A.shape[2],
                       A.shape[1] * A.shape[2], tB, B.shape[2], B.shape[1] * B.shape[2], beta, out.ptr, out.ldc,
                       out.M * out.ldc, sh.batch)
    torch.cuda.synchronize()
    assert lib.device_status() == 0
    return out.result(sh.N)


# Edges of the tiles (rows of 128 and 256, columns of 64, 128 and 256), one more and one
# less; K below, at and past one chunk and the ring's chunks; more tiles than CTAs; splits
# with a short last range; rows that allow 32-byte, 16-byte and 4-byte access only.
CASES = [(1, 1, 1, 1, 1, 1), (127, 65, 31, 1, 4, 1), (129, 255, 33, 2, 1, 1), (256, 256, 32, 1, 8, 1),
         (257, 130, 96, 2, 4, 1), (300, 513, 300, 1, 1, 3), (64, 64, 1000, 3, 8, 16), (2000, 1500, 65, 2, 4, 1)]


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("trans", ["NN", "NT", "TN", "TT"])
def test_against_oracle(lib, torch, bn, trans):
    for i, (M, N, K, batch, pad, splits) in enumerate(CASES):
        sh = wl.Shape(M, N, K, batch, trans[0], trans[1])
        beta = 0.5 if i % 2 else 0.0
        A, B, C0 = wl.gemm_inputs(sh, seed=100 + i, ld_multiple=pad, beta_nonzero=beta != 0)
        got = run(lib, torch, bn, splits, sh, A, B, C0, -1.5, beta)
        ref, den = og.gemm(sh.transA, sh.transB, M, N, K, -1.5, A, B, beta, C0 if beta else None,
                           nthreads=og.max_threads())
        assert og.error_ratio(got, ref, den) <= tolerance(K, splits), sh


@pytest.mark.parametrize("bn", [64, 128, 256])
def test_integers_exact_and_splits_repeatable(lib, torch, bn):
    sh = wl.Shape(270, 200, 700, 2, "N", "N")
    A, B, C0 = wl.gemm_inputs(sh, seed=7, kind="integer", bound=100)
    ref, _ = og.gemm("N", "N", sh.M, sh.N, sh.K, 1.0, A, B)
    for splits in (1, 4):
        first = run(lib, torch, bn, splits, sh, A, B, C0, 1.0, 0.0)
        assert np.array_equal(first.astype(np.float64), ref)
        assert np.array_equal(first, run(lib, torch, bn, splits, sh, A, B, C0, 1.0, 0.0))


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("kind", ["inf", "nan", "overflow", "tiny", "denormal", "zero", "products"])
def test_values_that_do_not_split(lib, torch, bn, kind):
    """Infinities, NaN, values that round past the largest BF16 and values whose low bits
    are below BF16's range give what the FP32 FMAs of the SIMT family give."""
    sh = wl.Shape(300, 280, 150, 1, "N", "T")
    A, B, C0 = wl.gemm_inputs(sh, seed=3)
    if kind == "inf":
        A[0, 140, 77] = np.inf
    elif kind == "nan":
        B[0, 200, 3] = np.nan
    elif kind == "overflow":
        A[0, 5, :sh.K] = 3.4e38
        B[0, 6, :sh.K] = np.abs(B[0, 6, :sh.K])
    elif kind == "tiny":
        A[:, :, :sh.K] *= np.float32(2.0 ** -118)
    elif kind == "denormal":
        B[0, 9, :sh.K] *= np.float32(2.0 ** -140)
    elif kind == "products":  # every factor splits, every product is denormal
        A[:, :, :sh.K] *= np.float32(2.0 ** -70)
        B[:, :, :sh.K] *= np.float32(2.0 ** -66)
    else:
        A[:, :, :sh.K] = 0
        B[0, 17, :sh.K] = -0.0
    got = run(lib, torch, bn, 1, sh, A, B, C0, 1.0, 0.0)[0]
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    out = Out(torch, C0, 0.0, sh.N)
    lib.gemm_with_config(533, "N", "T", sh.M, sh.N, sh.K, 1.0, tA, A.shape[2], tB, B.shape[2], 0.0, out.ptr, out.ldc, 1)
    torch.cuda.synchronize()
    want = out.result(sh.N)[0]
    assert np.array_equal(np.isnan(got), np.isnan(want))
    odd = ~np.isfinite(want)
    assert np.array_equal(got[odd & ~np.isnan(want)], want[odd & ~np.isnan(want)])
    a, b = A[0, :, :sh.K].astype(np.float64), B[0, :, :sh.K].astype(np.float64)
    with np.errstate(invalid="ignore", over="ignore"):
        ref, den = a @ b.T, np.abs(a) @ np.abs(b).T
    ok = np.isfinite(want)
    # FMA chains of K terms, and results that are denormal themselves
    assert np.all(np.abs(got - ref)[ok] <= (sh.K + 2) * 2.0 ** -24 * den[ok] + sh.K * 2.0 ** -149)


@pytest.mark.parametrize("trans", ["NN", "NT", "TN", "TT"])
@pytest.mark.parametrize("bn,pad", [(64, 1), (128, 4), (256, 8), (256, 1)])
def test_computed_again_in_every_layout(lib, torch, trans, bn, pad):
    """Every tile by FMAs: each row of A holds a value whose low bits are below BF16's range."""
    sh = wl.Shape(275, 261, 70, 2, trans[0], trans[1])
    A, B, C0 = wl.gemm_inputs(sh, seed=11, ld_multiple=pad, beta_nonzero=True)
    if trans[0] == "N":
        A[:, :, 33] = np.float32(1.2345e-36)
    else:
        A[:, 33, :sh.M] = np.float32(1.2345e-36)
    for splits in (1, 2):
        got = run(lib, torch, bn, splits, sh, A, B, C0, 2.0, 0.5)
        ref, den = og.gemm(sh.transA, sh.transB, sh.M, sh.N, sh.K, 2.0, A, B, 0.5, C0)
        assert og.error_ratio(got, ref, den) <= (sh.K + 4) * 2.0 ** -24


def test_shared_operand_strides(lib, torch):
    """A zero batch stride (one matrix for every entry) and gapped operands."""
    M, N, K, batch = 140, 170, 90, 3
    rng = np.random.default_rng(0)
    A = rng.uniform(-1, 1, (M, K)).astype(np.float32)
    B = rng.uniform(-1, 1, (batch, K + 2, N + 2)).astype(np.float32)
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.full((batch, M + 1, N), float("nan"), device="cuda")
    for bn in (64, 128, 256):
        lib.f32tc_selftest(bn, 1, "N", "N", M, N, K, 1.0, tA, K, 0, tB, N + 2, (K + 2) * (N + 2), 0.0, C, N,
                           (M + 1) * N, batch)
        got = C.cpu().numpy()
        for b in range(batch):
            ref, den = og.gemm("N", "N", M, N, K, 1.0, A[None], B[b:b + 1, :K])
            assert og.error_ratio(got[b:b + 1, :M], ref, den) <= tolerance(K, 1)
        assert np.all(np.isnan(got[:, M]))


def test_no_less_exact_than_simt(lib, torch):
    """Where a handle call uses the tensor cores, the error against 64 bits is at most the
    selected SIMT kernel's, on signed and on non-negative data, over the range of K."""
    h = lib.Handle(json.load(open(os.path.join(DEPLOY, "f32.json"))))
    used = 0
    for i, (M, N, K) in enumerate([(700, 650, 4096), (1500, 2200, 128), (1024, 1024, 700), (2048, 3024, 96),
                                   (333, 3000, 2000)]):
        for lo in (-1.0, 0.0):
            g = torch.Generator("cuda").manual_seed(i)
            A = torch.rand((M, K), generator=g, device="cuda") * (1 - lo) + lo
            B = torch.rand((K, N), generator=g, device="cuda") * (1 - lo) + lo
            cid = lib.select_kernel(h, M, N, K)
            used += lib.f32tc_choice(cid, M, N, K)[0] != 0
            ref = A.double() @ B.double()
            C = torch.empty((2, M, N), device="cuda")
            lib.gemm(h, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C[0], N)
            lib.gemm_with_config(cid, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C[1], N)
            err = [float((c.double() - ref).norm() / ref.norm()) for c in C]
            assert err[0] <= err[1], (M, N, K, lo, err)
    assert used >= 6


def test_handle_calls_under_capture(lib, torch):
    """A split tensor-core product through gemm(), eager and replayed from a CUDA graph: the same bits."""
    h = lib.Handle(json.load(open(os.path.join(DEPLOY, "f32.json"))))
    M, N, K = 512, 384, 4096
    bn, splits = lib.f32tc_choice(lib.select_kernel(h, M, N, K), M, N, K)
    assert bn and splits > 1
    A, B = torch.rand((M, K), device="cuda"), torch.rand((K, N), device="cuda")
    C = torch.empty((M, N), device="cuda")
    lib.gemm(h, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C, N)
    torch.cuda.synchronize()
    eager = C.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        lib.gemm(h, "N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C, N)
    C.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(C, eager)
