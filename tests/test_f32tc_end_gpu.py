"""The end of the FP32 tensor-core kernels: each CTA waits for the arrivals that free its
ring's last slots, for fewer, as many and more chunks than the ring has, and for CTAs with
one item and several; back to back, so that a CTA follows another on its SM.  Integer
products, which are exact."""
import numpy as np
import pytest

from oracle import gemm as og
from paper_2008_13145_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("K", [32, 64, 96, 128, 160, 257])  # 1 .. 5 and 9 chunks; rings of 3 and 4
@pytest.mark.parametrize("M,N", [(260, 130), (2100, 2600)])
def test_launches_in_a_row(lib, bn, K, M, N):
    import torch
    sh = wl.Shape(M, N, K, 1, "N", "T")
    A, B, _ = wl.gemm_inputs(sh, seed=K, kind="integer", bound=100)
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.full((20, M, N), float("nan"), device="cuda")
    for i in range(20):
        lib.f32tc_selftest(bn, 1, "N", "T", M, N, K, 1.0, tA, A.shape[2], 0, tB, B.shape[2], 0, 0.0, C[i], N, 0)
    torch.cuda.synchronize()
    assert lib.device_status() == 0
    ref, _ = og.gemm("N", "T", M, N, K, 1.0, A, B, nthreads=og.max_threads())
    want = torch.from_numpy(ref[0]).cuda()
    assert all(torch.equal(c.double(), want) for c in C)
