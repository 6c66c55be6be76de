"""Linear combinations of a matrix with its own transpose (one pass over tile
pairs) and scalars +-2^k (exponent arithmetic instead of multiplies): the bits
of the general kernels and of the multiplication."""
import pytest
import torch

import bq_inputs as bi
import paper_2609_02081_gb300 as hm

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with hm.Handle() as h:
        yield h


@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 100])
@pytest.mark.parametrize("opA,opB", [("N", "H"), ("H", "N"), ("C", "T"), ("T", "QC")])
def test_pair_kernel_gives_the_general_kernels_bits(handle, n, opA, opB):
    """op(X) + op'(X) with one transposing op: the same as with a copy of X as the second operand (which takes the
    general kernel), for every kind of scalar, flags that differ, and a strided X whose absent component is NaN."""
    X = bi.uniform(900 + n, n, n + 3).to(DEV)[:, :, :n]
    X[0, 0, 0] = 0.0
    special = torch.tensor([5e-324, -2.3e-308, 3e-300, 1.7e308, float("inf"), 1e-270, -0.0, 1e-275], dtype=torch.float64)
    X[:, n // 2, n // 3] = special.to(DEV)
    X[:, n // 3, n // 2] = special.flip(0).to(DEV)
    for fa, fb in ((0xFF, 0xFF), (0x7F, 0xF7)):
        if fa != 0xFF:
            X = X.clone()
        Y = X.clone()
        for al, be in ((0.5, 0.5), (1.0, 1.0), (-0.25, 2.0), (0.25, -0.25), (-2.0 ** -32, 2.0 ** -32), (1j, 0.3), (1.5 - 0.5j, -1j), (4.0, -1.0)):
            got = torch.full((8, n, n), float("nan"), dtype=torch.float64, device=DEV)
            want = got.clone()
            hm.hmat_bq_add(handle, X, X, got, al, be, opA, opB, fa, fb)
            hm.hmat_bq_add(handle, X, Y, want, al, be, opA, opB, fa, fb)
            torch.cuda.synchronize()
            nan = torch.isnan(want)
            assert torch.equal(torch.isnan(got), nan)
            assert torch.equal(got[~nan].view(torch.int64), want[~nan].view(torch.int64)), (al, be)


@pytest.mark.parametrize("k", [-64, -2, -1, 1, 3, 64])
def test_power_of_two_scalars_are_exact_products(handle, k):
    """x 2^k for zeros, subnormals, the range's ends, infinities and NaN, in rows and in transposed tiles: the bits of
    the rounded product (a NaN stays one)."""
    vals = [0.0, -0.0, 5e-324, -3e-320, 2.2250738585072014e-308, 4.4e-308, 1e-290, -1.0, 3.0, 1e300, 8.9e307,
            1.7976931348623157e308, float("inf"), float("-inf"), float("nan"), -1e-5]
    n = 37
    X = torch.tensor(vals, dtype=torch.float64).repeat(8 * n * n // len(vals) + 1)[:8 * n * n].view(8, n, n).to(DEV)
    for s in (2.0 ** k, -(2.0 ** k)):
        want = X * s
        for op, ref in (("N", want), ("T", want.transpose(1, 2))):
            sign = torch.tensor([1, 1, -1, 1, 1, 1, -1, 1], dtype=torch.float64, device=DEV).view(8, 1, 1)
            ref = ref * sign if op == "T" else ref
            Y = torch.empty((8, n, n), dtype=torch.float64, device=DEV)
            Z = torch.zeros((8, n, n), dtype=torch.float64, device=DEV)
            hm.hmat_bq_add(handle, X, Z, Y, s, 1.0, op, "N")      # + 0: turns -0 to +0
            ref = ref + 0.0
            torch.cuda.synchronize()
            nan = torch.isnan(ref)
            assert torch.equal(torch.isnan(Y), nan)
            assert torch.equal(Y[~nan].view(torch.int64), ref[~nan].view(torch.int64))
