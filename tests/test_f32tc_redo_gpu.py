"""Tiles that the FP32 products on the tensor cores compute again by FMAs, because an
operand does not split or an accumulator overflowed: where they lie among a CTA's
items, at long K, through handle calls, and what they cost."""
import json
import os

import pytest

from tests.test_f32tc_gpu import DEPLOY

pytestmark = pytest.mark.gpu
TINY = 1.2345e-36  # its low bits are below BF16's range: such a value does not split


@pytest.fixture(scope="module")
def torch():
    import torch as t
    return t


@pytest.fixture(scope="module")
def handle(lib):
    return lib.Handle(json.load(open(os.path.join(DEPLOY, "f32.json"))))


def uniform(torch, seed, *shape):
    return torch.rand(shape, generator=torch.Generator("cuda").manual_seed(seed), device="cuda") * 2 - 1


def check(torch, got, A, B, C0=None, beta=0.0):
    """NaN where the exact product has it, else within a K-term FMA chain's bound.  Where the absolute
    values sum past FP32's range a chain may overflow on the way, in any order: not compared."""
    a, b = A.double(), B.double()
    ref, den = a @ b, a.nan_to_num(0, 0, 0).abs() @ b.nan_to_num(0, 0, 0).abs()
    if beta:
        ref, den = ref + beta * C0.double(), den + abs(beta) * C0.double().abs()
    in_range = den <= torch.finfo(torch.float32).max
    assert torch.equal(got[in_range].isnan(), ref[in_range].isnan())
    odd = ref.isinf()
    assert torch.equal(got[odd].double(), ref[odd])
    ok = ref.isfinite() & in_range
    assert bool(((got.double() - ref).abs()[ok] <= (A.shape[1] + 4) * 2.0 ** -24 * den[ok] + 2.0 ** -149).all())


# Every tile width that a handle call chooses here, whole and with K divided.
@pytest.mark.parametrize("M,N,K", [(2048, 2048, 512), (1433, 1100, 1003), (512, 384, 4096), (323, 3000, 700)])
@pytest.mark.parametrize("kind", ["nan", "inf", "tiny rows", "tiny column", "overflow"])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_through_handle_calls(lib, torch, handle, M, N, K, kind, beta):
    assert lib.f32tc_choice(lib.select_kernel(handle, M, N, K), M, N, K, aligned=N % 4 == 0 and K % 4 == 0)[0]
    A, B, C0 = uniform(torch, 1, M, K), uniform(torch, 2, K, N), uniform(torch, 3, M, N)
    if kind == "nan":
        A[M - 1, K - 1] = float("nan")
    elif kind == "inf":
        B[K // 2, N - 1] = float("inf")
    elif kind == "tiny rows":
        A[:, 5] = TINY
    elif kind == "tiny column":
        B[:, 33] *= TINY
    else:
        A[7], B[:, 9] = 3e38, B[:, 9].abs()
    C = C0.clone()
    lib.gemm(handle, "N", "N", M, N, K, 1.0, A, K, B, N, beta, C, N)
    torch.cuda.synchronize()
    assert lib.device_status() == 0
    check(torch, C, A, B, C0, beta)


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("transA,transB", ["NT", "TN"])
def test_longest_k(lib, torch, bn, transA, transB):
    """K = 2^18, the longest that the kernels take, in one item: no wait runs out while its tile is computed again."""
    M, N, K = 130, 70, 1 << 18
    A, B = uniform(torch, 4, M, K), uniform(torch, 5, K, N)
    A[128, 1000] = float("nan")
    A[3, 70000] = TINY
    sA = A if transA == "N" else A.t().contiguous()
    sB = B if transB == "N" else B.t().contiguous()
    C = torch.zeros((M, N), device="cuda")
    lib.f32tc_selftest(bn, 1, transA, transB, M, N, K, 1.0, sA, sA.shape[1], 0, sB, sB.shape[1], 0, 0.0, C, N, 0)
    torch.cuda.synchronize()
    assert lib.device_status() == 0
    check(torch, C, A, B)


# Items of 128 rows x 1 column: 1,020 to a CTA on 152 SMs, the most (1,024) and two CTAs' worth.
@pytest.mark.parametrize("rows", [128 * 155040, 128 * 155648, 128 * 155649 + 1])
def test_marks_of_many_items(lib, torch, rows):
    A = uniform(torch, 6, rows, 1)
    for at in (0, 1, 128, 127 + 128 * 152 * 3, rows // 2, rows - 130, rows - 1):
        A[at] = TINY
    b = torch.full((1, 1), 1.5, device="cuda")
    C = torch.full((rows, 1), float("nan"), device="cuda")
    lib.f32tc_selftest(64, 1, "N", "N", rows, 1, 1, 1.0, A, 1, 0, b, 1, 0, 0.0, C, 1, 0)
    want = A.double() * 1.5
    # a product rounded once, or truncated in the accumulator
    assert bool(((C.double() - want).abs() <= 2.0 ** -22 * want.abs()).all())
    assert lib.device_status() == 0


@pytest.mark.parametrize("where", ["A", "B"])
def test_one_nan_costs_no_more_than_twice_the_selected_kernel(lib, torch, handle, where):
    n = 2048
    cid = lib.select_kernel(handle, n, n, n)
    assert lib.f32tc_choice(cid, n, n, n)[0]
    A, B, C = uniform(torch, 7, n, n), uniform(torch, 8, n, n), torch.empty((n, n), device="cuda")
    (A if where == "A" else B)[1000, 700] = float("nan")

    def fastest(call):
        times = []
        for _ in range(8):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            call()
            t1.record()
            t1.synchronize()
            times.append(t0.elapsed_time(t1))
        return min(times[3:])

    simt = fastest(lambda: lib.gemm_with_config(cid, "N", "N", n, n, n, 1.0, A, n, B, n, 0.0, C, n))
    assert fastest(lambda: lib.gemm(handle, "N", "N", n, n, n, 1.0, A, n, B, n, 0.0, C, n)) <= 2 * simt
