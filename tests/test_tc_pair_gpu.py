"""The 256 x 256 tiles of CTA pairs, which the BN 256 configs use past 128 rows: integer
products, which the tensor cores sum exactly, at the edges of the tiles and of a K slice."""
import numpy as np
import pytest

from oracle import gemm as og
from paper_2008_13145_gb300 import workloads as wl
from tests.gpu_helpers import Out

pytestmark = pytest.mark.gpu

# One row in the second CTA's half; a whole tile; one more each way; a tile whose second
# half of columns is empty; more K slices than stages with a short last one; several
# tiles a pair (76 pairs); rows of C that allow 32-, 16- and 4-byte access.
CASES = [(129, 8, 16, 1, 8), (256, 256, 64, 1, 8), (257, 260, 72, 2, 4), (300, 100, 1000, 1, 1),
         (511, 300, 450, 1, 4), (2000, 700, 96, 4, 8)]


@pytest.mark.parametrize("cid", [1016, 1116, 1216])
@pytest.mark.parametrize("trans", ["NN", "NT", "TN", "TT"])
def test_integer_products(lib, cid, trans):
    import torch
    for i, (M, N, K, batch, pad) in enumerate(CASES):
        sh = wl.Shape(M, N, K, batch, trans[0], trans[1])
        A, B, C0 = wl.gemm_inputs(sh, seed=40 + i, ld_multiple=pad, beta_nonzero=True, kind="integer", bound=8)
        beta = float(i % 2)
        tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
        if cid // 100 == 11:
            tA, tB = tA.to(torch.bfloat16), tB.to(torch.bfloat16)
        out = Out(torch, C0, beta, N)
        lib.gemm_with_config(cid, trans[0], trans[1], M, N, K, 2.0, tA, A.shape[2], tB, B.shape[2], beta, out.ptr,
                             out.ldc, batch)
        torch.cuda.synchronize()
        assert lib.device_status() == 0
        ref, _ = og.gemm(trans[0], trans[1], M, N, K, 2.0, A, B, beta, C0, nthreads=og.max_threads())
        assert np.array_equal(out.result(N).astype(np.float64), ref), (cid, sh)
