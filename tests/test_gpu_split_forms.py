"""Split mode's forms where the tests of one form do not reach the others: modulus counts
that mix in one launch, the largest outputs of each form's own moduli, the deepest products, the
no-allocation entry point."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

import bq_inputs as bi
import oracle
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


def product_tensor():
    """T[e, c, d]: output component e of the product of storage basis elements c and d (oracle)."""
    eye = np.eye(8)
    return np.array([[oracle.bq_gemm(eye[c].reshape(8, 1, 1), eye[d].reshape(8, 1, 1))[:, 0, 0] for d in range(8)]
                     for c in range(8)]).transpose(2, 0, 1)


@pytest.mark.parametrize("form,tol,k,count", [("gauss", 1e-12, 11854, 14), ("gauss", 1e-13, 8937, 15),
                                              ("gauss", 1e-14, 106689, 16), ("auto", 1e-12, 290, 14),
                                              ("auto", 1e-12, 29349, 15), ("auto", 1e-13, 11120, 16),
                                              ("auto", 1e-14, 61858, 17)])
def test_largest_outputs_of_each_forms_moduli(handles, form, tol, k, count):
    """Each form at the margin of its own moduli: the largest k that `count` of them serve, every
    entry +-(2 - 2^-40) with the signs that make one component the sum of all its 8 k terms, so
    that |Q| is within 0.25 % of the P / 2^1.25 from which the CRT's quotient is still taken as
    the nearest integer.  The output is k N c^2 with integers N, rounded once."""
    bits = hm.split_info(k, tol)[1]
    moduli = hm.split_info(k, tol)[0] if form == "gauss" else MATRIX_MODULI[:matrix_form_moduli(k, tol)]
    assert len(moduli) == count
    largest = 8 * k * (2 ** bits - 2 ** (bits - 41)) ** 2
    assert 0.9975 / 2 ** 1.25 < largest / math.prod(int(p) for p in moduli) < 1 / 2 ** 1.25
    signs = np.array([[1.0 if (v >> c) & 1 else -1.0 for c in range(8)] for v in range(256)])
    Q = np.einsum("sc,ecd,td->est", signs, product_tensor(), signs)
    e, sa, sb = np.unravel_index(np.argmax(np.abs(Q)), Q.shape)
    N = Q[:, sa, sb]
    assert abs(N[e]) == 8.0
    c, (m, n) = 2.0 - 2.0 ** -40, (3, 5)
    A = torch.from_numpy(signs[sa] * c).cuda()[:, None, None].expand(8, m, k).contiguous()
    B = torch.from_numpy(signs[sb] * c).cuda()[:, None, None].expand(8, k, n).contiguous()
    want = np.array([float(Fraction(int(v) * k) * Fraction(c) ** 2) for v in N])
    for sign in (1.0, -1.0):
        C = torch.full((8, m, n), float("nan"), dtype=torch.float64, device="cuda")
        hm.hmat_bq_gemm(handles[form], sign * A, B, C, mode="split", tol=tol)
        np.testing.assert_array_equal(C.cpu().numpy(), np.broadcast_to((sign * want)[:, None, None], (8, m, n)))


def test_deepest_four_multiplication_products(handles):
    """The forced four-multiplication form runs over 2 k: at the largest k 254 accumulation chunks,
    whose running sums stay below 2^15: Gauss's and the default form's bits."""
    k, m, n = 127 * 1024, 20, 40
    A, B = bi.uniform(530, m, k).cuda(), bi.uniform(531, k, n).cuda()
    outs = []
    for form in ("four_m", "gauss", "auto"):
        C = torch.full((8, m, n), float("nan"), dtype=torch.float64, device="cuda")
        hm.hmat_bq_gemm(handles[form], A, B, C, mode="split", tol=1e-12)
        outs.append(C)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[2], outs[1])


@pytest.mark.parametrize("m,n,k", [(96, 112, 200), (33, 20, 600)])
def test_noalloc_in_the_four_multiplication_form(handles, m, n, k):
    """The no-allocation entry point with that form forced, one accumulation chunk and several of
    its doubled depth: the workspace path's bits, and twice in a row."""
    h = handles["four_m"]
    A, B = bi.fock_like(540, m, k, row_scale=True).cuda(), bi.uniform(541, k, n).cuda()
    C0 = bi.uniform(542, m, n).cuda()
    want = C0.clone()
    hm.hmat_bq_gemm(h, A, B, want, alpha=0.5 - 2j, beta=1.5 + 0.25j, mode="split", tol=1e-12)
    for _ in range(2):
        got = C0.clone()
        hm.hmat_bq_gemm_split_noalloc(h, A, B, got, alpha=0.5 - 2j, beta=1.5 + 0.25j, tol=1e-12)
        torch.cuda.synchronize()
        assert torch.equal(got, want)
