"""The single-CTA and the grouped tensor-core kernels where a warp's last rows of C do not
exist and every row allows 32-byte stores (the other lanes go past M): integer products,
which the tensor cores sum exactly, several 32-column chunks and tiles a warp."""
import numpy as np
import pytest

from oracle import gemm as og
from paper_2008_13145_gb300 import workloads as wl
from tests.gpu_helpers import Out

pytestmark = pytest.mark.gpu

# M: one row, one more and one less than a warp's 32 and a tile's 128; BN 256 past 128 rows
# runs on CTA pairs, so its cases keep to 128.
ROWS = (1, 31, 33, 97, 127, 129, 161, 257)


def operands(torch, sh, seed, bf16):
    A, B, C0 = wl.gemm_inputs(sh, seed=seed, ld_multiple=8, beta_nonzero=True, kind="integer", bound=8)
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    return (A, B, C0), (tA.to(torch.bfloat16), tB.to(torch.bfloat16)) if bf16 else (tA, tB)


@pytest.mark.parametrize("family", [1, 2, 3])
@pytest.mark.parametrize("bn_slot", [0, 1, 2])
def test_single_cta(lib, family, bn_slot):
    import torch
    cid = lib.config_ids(family)[3 * bn_slot]
    for i, M in enumerate(m for m in ROWS if bn_slot < 2 or m <= 128):
        sh = wl.Shape(M, 520, 200, 3, "N", "T")
        (A, B, C0), (tA, tB) = operands(torch, sh, i, family == 2)
        beta = float(i % 2)
        out = Out(torch, C0, beta, sh.N)
        lib.gemm_with_config(cid, "N", "T", M, sh.N, sh.K, 2.0, tA, A.shape[2], tB, B.shape[2], beta, out.ptr, out.ldc, 3)
        torch.cuda.synchronize()
        assert lib.device_status() == 0
        ref, _ = og.gemm("N", "T", M, sh.N, sh.K, 2.0, A, B, beta, C0)
        assert np.array_equal(out.result(sh.N).astype(np.float64), ref), (cid, M)


@pytest.mark.parametrize("family", [1, 2, 3])
@pytest.mark.parametrize("bn_slot", [0, 1, 2])
def test_grouped(lib, family, bn_slot):
    import torch
    cid = lib.config_ids(family)[3 * bn_slot]
    probs, want = [], []
    for i, M in enumerate(ROWS):
        sh = wl.Shape(M, 264 + 32 * i, 72 + 8 * i, 1, "N", "T")
        (A, B, C0), (tA, tB) = operands(torch, sh, 10 + i, family == 2)
        C = torch.from_numpy(np.nan_to_num(C0, nan=0.0)).cuda()
        probs.append(dict(M=M, N=sh.N, K=sh.K, transA="N", transB="T", alpha=1.0, beta=float(i % 2), A=tA,
                          lda=A.shape[2], B=tB, ldb=B.shape[2], C=C, ldc=C0.shape[2]))
        want.append(og.gemm("N", "T", M, sh.N, sh.K, 1.0, A, B, float(i % 2), C0)[0][0])
    lib.gemm_grouped_with_config(cid, probs)
    torch.cuda.synchronize()
    assert lib.device_status() == 0
    for q, ref in zip(probs, want):
        assert np.array_equal(q["C"].cpu().numpy()[0, :, :q["N"]].astype(np.float64), ref), (cid, q["M"])
