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


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("shapes", [
    [(256, 256, 256)],                                       # ranges that cross tiles
    [(33, 32, 32)],                                          # the shortest k that is cut
    [(64, 64, 131)],                                         # pieces within a tile, a ragged last one
    [(32, 32, 2001)],                                        # one tile on every SM
    [(250, 200, 300), (64, 40, 0), (33, 40, 1000), (10, 9, 50)]])
def test_fp64_ranges(shapes, use_graph):
    """Calls of few tiles are cut into equal ranges of the inner dimension when the workspace
    holds the partial tiles, into fewer slices or none when it is smaller: the same exact result
    with complex alpha and beta, also for a product without an inner dimension."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    alpha, beta = 1 - 2j, 2 + 1j
    with hm.Handle() as h:
        probs = []
        for i, (m, n, k) in enumerate(shapes):
            fb = bi.TRA if i == 2 else bi.BQ
            A, B, C0 = bi.small_int(700 + i, m, k), bi.small_int(710 + i, k, n, flags=fb), bi.small_int(720 + i, m, n)
            probs.append((A.cuda(), B.cuda(), torch.empty_like(C0, device="cuda"), C0, fb,
                          oracle.bq_gemm(A.numpy(), B.numpy(), alpha=alpha, beta=beta, C=C0.numpy())))
        descs = [hm.make_desc(a, b, c, flagsB=fb, alpha=alpha, beta=beta) for a, b, c, _, fb, _ in probs]
        need = hm.hmat_workspace_size(h, descs, "fp64")
        assert need > 0
        s = torch.cuda.Stream()
        for size in (need, need - 1, 4 << 20, 256):
            ws = torch.empty(size, dtype=torch.uint8, device="cuda")
            for _, _, c, c0, _, _ in probs:
                c.copy_(c0)
            torch.cuda.synchronize()
            hm.hmat_bq_gemm_grouped(h, descs, "fp64", workspace=ws, use_graph=use_graph, stream=s)
            torch.cuda.synchronize()
            for _, _, c, _, _, want in probs:
                np.testing.assert_array_equal(c.cpu().numpy(), want)
        assert h.device_error() == 0
