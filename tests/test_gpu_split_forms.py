"""Split mode's forms where the tests of one form do not reach the others: modulus counts
that mix in one launch."""
import math

import pytest
import torch

import bq_inputs as bi
import paper_2609_02081_gb300 as hm
from test_mat2_form import MODULI as MATRIX_MODULI

pytestmark = pytest.mark.gpu


@pytest.fixture
def handles():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    made = {form: hm.Handle() for form in ("auto", "gauss", "four_m")}
    for form, h in made.items():
        h.set_complex_form(form)
    yield made
    for h in made.values():
        assert h.device_error() == 0
        h.close()


def matrix_form_moduli(k, tol):
    """Modulus count of the matrix form: P above 2^0.25 times twice the largest output, 8 k 2^(2 bits)."""
    bits = hm.split_info(k, tol)[1]
    n = 0
    while math.log2(math.prod(MATRIX_MODULI[:n])) <= 2 * bits + math.log2(k) + 4.25:
        n += 1
    return n


@pytest.mark.parametrize("tol,ks,counts", [(1e-13, (1, 64, 114, 115, 300), (14, 15, 15, 16, 16)),
                                           (1e-14, (7, 8, 200, 695, 696), (15, 16, 16, 16, 17))])
@pytest.mark.parametrize("use_graph", [False, True])
def test_modulus_counts_mixed_in_one_launch(handles, tol, ks, counts, use_graph):
    """Jobs of up to 15 moduli (whose CRT tables are scaled to fill four limbs) beside jobs of more
    run in the five-limb kernel together: the bits of an all-Gauss handle, each flag pair."""
    assert tuple(matrix_form_moduli(k, tol) for k in ks) == counts
    pairs = [(bi.BQ, bi.BQ), (bi.TRS, bi.TRA), (bi.COMPLEX, bi.BQ), (bi.COMPLEX, bi.COMPLEX), (bi.BQ, bi.TRS)]
    probs = []
    for i, k in enumerate(ks):
        for j, (fa, fb) in enumerate(pairs):
            m, n = 5 + 31 * j, 33 + 17 * i
            probs.append((bi.fock_like(500 + i, m, k, row_scale=True).cuda(), bi.uniform(510 + j, k, n).cuda(), fa, fb))
    res = []
    for form in ("auto", "gauss"):
        outs = [torch.full((8, a.shape[1], b.shape[2]), float("nan"), dtype=torch.float64, device="cuda")
                for a, b, _, _ in probs]
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        descs = [hm.make_desc(a, b, c, flagsA=fa, flagsB=fb, alpha=0.5 - 2j) for (a, b, fa, fb), c in zip(probs, outs)]
        ws = torch.empty(hm.hmat_workspace_size(handles[form], descs, "split", tol), dtype=torch.uint8, device="cuda")
        hm.hmat_bq_gemm_grouped(handles[form], descs, "split", tol, ws, s, use_graph)
        s.synchronize()
        res.append(outs)
    for (a, b, fa, fb), got, want in zip(probs, *res):
        assert torch.equal(got, want), (a.shape, b.shape, fa, fb)
