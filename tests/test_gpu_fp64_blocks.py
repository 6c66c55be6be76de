"""FP64 mode around the edges of the kernel's k-blocks (4 wide, staged two ahead) and
32 x 32 tiles: on small integers every factor, product and sum is exact, so the
result equals the oracle's bits."""
import numpy as np
import pytest
import torch

import bq_inputs as bi
import oracle
import paper_2609_02081_gb300 as hm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(1, 1), (31, 33), (64, 32)])
@pytest.mark.parametrize("opA,opB,fa,fb", [("N", "N", bi.BQ, bi.BQ), ("H", "T", bi.BQ, bi.TRA),
                                           ("QC", "C", bi.COMPLEX, bi.BQ), ("T", "H", bi.TRS, bi.TRS)])
def test_fp64_k_blocks(m, n, opA, opB, fa, fb):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with hm.Handle() as h:
        for k in (1, 2, 3, 4, 5, 7, 8, 9, 11, 12, 13, 16, 37):
            A = bi.small_int(600 + k, *((k, m) if opA in ("T", "H") else (m, k)), flags=fa)
            B = bi.small_int(650 + k, *((n, k) if opB in ("T", "H") else (k, n)), flags=fb)
            C = torch.full((8, m, n), float("nan"), dtype=torch.float64, device="cuda")
            hm.hmat_bq_gemm(h, A.cuda(), B.cuda(), C, opA, opB, fa, fb, mode="fp64")
            torch.cuda.synchronize()
            np.testing.assert_array_equal(C.cpu().numpy(), oracle.bq_gemm(A.numpy(), B.numpy(), opA, opB))
        assert h.device_error() == 0
