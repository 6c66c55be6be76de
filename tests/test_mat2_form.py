"""The matrix form of split-mode products (split_mat2.cu).

Modulo p with s^2 = -1 the biquaternions are two copies of the 2 x 2 matrices;
each copy's product takes Winograd's seven multiplications.  The CPU tests
restate that algebra and the kernels' exact arithmetic on integers; the GPU
tests require the bits of Gauss's form, which computes the same exact integers
through the paper's products.
"""
import itertools
import math
import random

import numpy as np
import pytest
import torch

import bq_inputs as bi
import paper_2609_02081_gb300 as hm

MODULI = (241, 233, 229, 221, 205, 197, 193, 181, 173, 157, 149, 137, 113, 109, 101, 97, 89)
TOL = 1e-12


def centred(v, p):
    r = v % p
    return r - p if r > (p - 1) // 2 else r


def root(p):
    """The root of -1 with the smallest sum of digit weights, up to sign."""
    def weight(s):
        return sum(abs(centred(1 << (16 * d), p)) + abs(centred(s << (16 * d), p)) for d in range(3))
    return min((s for s in range(1, p) if (s * s + 1) % p == 0), key=weight)


def quaternion_product(a, b):
    """Eight real components (M_e + i M_{e+4} the coefficient of 1, i, j, k)."""
    q, r = [complex(0)] * 4, None
    A = [(a[e], a[e + 4]) for e in range(4)]
    B = [(b[e], b[e + 4]) for e in range(4)]

    def mul(x, y):
        return x[0] * y[0] - x[1] * y[1], x[0] * y[1] + x[1] * y[0]
    signs = [[(0, 0, 1), (1, 1, -1), (2, 2, -1), (3, 3, -1)], [(0, 1, 1), (1, 0, 1), (2, 3, 1), (3, 2, -1)],
             [(0, 2, 1), (2, 0, 1), (3, 1, 1), (1, 3, -1)], [(0, 3, 1), (3, 0, 1), (1, 2, 1), (2, 1, -1)]]
    out = [0] * 8
    for e, terms in enumerate(signs):
        for f, g, sg in terms:
            re, im = mul(A[f], B[g])
            out[e] += sg * re
            out[e + 4] += sg * im
    return out


def entries(x):
    """(Re, Im) of the matrix entries 11, 12, 21, 22 of a biquaternion with integer components."""
    return [(x[0] - x[5], x[4] + x[1]), (x[2] - x[7], x[6] + x[3]), (-x[2] - x[7], x[3] - x[6]),
            (x[0] + x[5], x[4] - x[1])]


def left(x11, x12, x21, x22):
    s1 = x21 + x22
    s2 = s1 - x11
    return [x11, x12, x12 - s2, x22, s1, s2, x11 - x21]


def right(y11, y12, y21, y22):
    t3 = y22 - y12
    t2 = t3 + y11
    return [y11, y21, y22, t2 - y21, y12 - y11, t2, t3]


def matrices(x, s, p):
    """The entries 11, 12, 21, 22 modulo p of both copies (the second one with -s for the coefficients' i)."""
    (r11, i11), (r12, i12), (r21, i21), (r22, i22) = entries(x)
    return ([(r + s * i) % p for r, i in entries(x)],
            [(r22 - s * i22) % p, (s * i21 - r21) % p, (s * i12 - r12) % p, (r11 - s * i11) % p])


def sums(t):
    """c11, c22, c12, c21 of the seven products."""
    u1 = t[0] + t[5]
    return [t[0] + t[1], u1 + t[6] + t[4], u1 + t[4] + t[2], u1 + t[6] - t[3]]


def contractands(u, v, half):
    """t11, t22, t12, t21 of a half from both copies' products."""
    cu, cv = sums(u), sums(v)
    cv = [cv[1], cv[0], -cv[3], -cv[2]]
    return [a - b if half else a + b for a, b in zip(cu, cv)]


def outputs(u, v):
    """The kernels' eight sums by (half, slot): 4 times (half 1: 4 s times) the component, modulo p."""
    out = {}
    for half in (0, 1):
        t11, t22, t12, t21 = contractands(u, v, half)
        z = [t11 + t22, t22 - t11, t12 - t21, -(t12 + t21)]
        for e in range(4):
            out[(4 * half + e) ^ ((e & 1) << 2)] = -z[e] if half and e & 1 else z[e]
    return out


def test_moduli_and_digit_weights():
    assert all(math.gcd(a, b) == 1 for a, b in itertools.combinations(MODULI, 2))
    assert all(p <= 255 and p % 2 == 1 for p in MODULI)
    for p in MODULI:
        s = root(p)
        assert (s * s + 1) % p == 0
        # u = sum_d x_d w_d + y_d s w_d over balanced 16-bit digits (the fourth below 2^6) is an exact float
        w = [abs(centred(1 << (16 * d), p)) + abs(centred(s << (16 * d), p)) for d in range(4)]
        assert sum(w[:3]) * (2 ** 15 + 1) + w[3] * 2 ** 6 < 2 ** 24
    # 1024-deep sums of products of residues up to 121 are exact in FP32
    assert 1024 * 121 ** 2 < 2 ** 24


def test_matrix_form_recombines_to_the_product():
    rng = random.Random(3)
    for p in MODULI:
        s = root(p)
        for _ in range(20):
            a, b = ([rng.randrange(-(1 << 46), (1 << 46) + 1) for _ in range(8)] for _ in range(2))
            copies = [[centred(f * g, p) for f, g in zip(left(*x), right(*y))]
                      for x, y in zip(matrices(a, s, p), matrices(b, s, p))]
            got = outputs(*copies)
            want = quaternion_product(a, b)
            for c in range(8):
                # half 1 (slots 0 and 2: imaginary parts of q1, q3; 1 and 3: real parts of q2, q4) carries s
                scale = 4 * s if c in (4, 1, 6, 3) else 4
                assert (got[c] - scale * want[c]) % p == 0, (p, c)
                assert abs(got[c]) <= 16 * (p - 1) // 2


def test_matrix_form_of_subalgebra_products():
    """A real quaternion's copies agree, so it is encoded once; one 2 x 2 product serves two of them (twice its sums
    stand for both copies' in the 1/4 and 1/(4 s) elements); a complex operand is one number per copy."""
    rng = random.Random(4)
    for p in MODULI:
        s = root(p)
        a, b, q = ([rng.randrange(-(1 << 46), (1 << 46) + 1) for _ in range(8)] for _ in range(3))
        a[4:] = q[4:] = [0] * 4
        x, y, z = matrices(a, s, p), matrices(b, s, p), matrices(q, s, p)
        assert x[0] == x[1]
        got = outputs(*[[centred(f * g, p) for f, g in zip(left(*x[0]), right(*yc))] for yc in y])
        want = quaternion_product(a, b)
        assert all((got[c] - (4 * s if c in (4, 1, 6, 3) else 4) * want[c]) % p == 0 for c in range(8))
        c11, c22, c12, c21 = sums([centred(f * g, p) for f, g in zip(left(*x[0]), right(*z[0]))])
        want = quaternion_product(a, q)
        for value, scale, w in ((c11 + c22, 4, want[0]), (c11 - c22, 4 * s, want[1]), (c12 - c21, 4, want[2]),
                                (c12 + c21, 4 * s, want[3])):
            assert (2 * value - scale * w) % p == 0
        c = [b[0], 0, 0, 0, b[4], 0, 0, 0]
        want = quaternion_product(c, q[:4] + b[4:])
        for e in range(4):
            u, v = (centred((c[0] + t * c[4]) * (q[e] + t * b[4 + e]), p) for t in (s, -s))
            assert (2 * (u + v) - 4 * want[e]) % p == 0 and (2 * (u - v) - 4 * s * want[e + 4]) % p == 0


def shift_of(nm):
    """Power of two by which the tables of up to 15 moduli are scaled: 2 N P just below 2^128."""
    if nm > 15:
        return 0
    return math.floor(127.99 - sum(math.log2(p) for p in MODULI[:nm]) - math.log2(2 * nm * 16 * 120))


def elements_of(nm, half):
    mods, P = MODULI[:nm], math.prod(MODULI[:nm])
    return [(P // p * (pow(P // p % p, -1, p) * pow(4 * root(p) if half else 4, -1, p) % p)) << shift_of(nm)
            for p in mods]


def test_mat2_crt_quotient_is_exact():
    """S = N P + sum_l x_l d_l with |x_l| <= 16 * 120 and N = nmod * 16 * 120: positive, within the limbs, and the
    float32 estimate of S / P rounds to the quotient for outputs up to |X| = P / 2^1.25: from the leading limb alone
    (up to 15 moduli, scaled to fill 128 bits), or from the limbs from the one below P's top."""
    W = 16 * 120
    rng = random.Random(12)
    for nm in range(1, len(MODULI) + 1):
        mods, sh = MODULI[:nm], shift_of(nm)
        P = math.prod(mods) << sh
        L = 4 if nm <= 15 else 5
        pb = max((P.bit_length() - 1) // 32 - 1, 0)
        pinv = np.float32(1.0 / sum(float((P >> (32 * q)) & 0xFFFFFFFF) * 2.0 ** (32 * (q - pb)) for q in range(pb, L)))
        assert 2 * nm * W * P < 2 ** (32 * L)
        lim = int((P >> sh) / 2 ** 1.25)
        for half in (0, 1):
            d = elements_of(nm, half)
            for trial in range(100):
                X = rng.choice([lim, -lim, rng.randrange(-lim, lim + 1), rng.randrange(-min(lim, 99), min(lim, 99) + 1)])
                S = nm * W * P
                for p, dl in zip(mods, d):
                    c = 4 * root(p) % p if half else 4
                    r = c * X % p
                    lo, hi = -W + (r + W) % p, W - (W - r) % p
                    S += rng.choice([lo, hi, lo + p * rng.randrange(0, (hi - lo) // p + 1)]) * dl
                assert 0 < S < 2 * nm * W * P
                limbs = [(S >> (32 * q)) & 0xFFFFFFFF for q in range(L)]
                sf = np.float32(limbs[L - 1])
                for q in range(L - 2, pb - 1, -1):
                    sf = np.float32(sf * np.float32(2.0 ** 32) + np.float32(limbs[q]))
                assert S - int(np.rint(np.float32(sf * pinv))) * P == X << sh, (nm, X)
                if nm <= 15:
                    q = int(np.rint(float(np.float32(limbs[3])) * float(np.float32(2.0 ** 96 / P))))
                    assert S - q * P == X << sh, (nm, X)


def test_mat2_crt_digit_sums():
    """The CRT's contraction restated: residues stored with 128 added, the sums c11, c22, c12, c21 of both copies (at
    most 2048, exact in FP16), u + v and u - v times the balanced 8-bit digits of the CRT elements, sums below 2^22,
    packed in pairs below 2^31; together with an offset less 128 times the weights they give N P + sum_l x_l d_l."""
    rng = random.Random(13)
    weights = {0: (1536, 0, 512, 0), 1: (0, -512, 0, 1536)}
    for nm in (1, 2, 14, 15, 16, 17):
        mods = MODULI[:nm]
        P = math.prod(mods) << shift_of(nm)
        for half in (0, 1):
            elements, digits = elements_of(nm, half), []
            for e in elements:
                dl = []
                for _ in range(17):
                    v = (e + 128) % 256 - 128
                    dl.append(v)
                    e = (e - v) >> 8
                assert e == 0 and dl[16] == 0
                digits.append(dl[:16])
            for i in range(16):
                worst = sum(abs(dl[i]) * 8 * ((p - 1) // 2 + 128) for dl, p in zip(digits, mods))
                assert worst < 2 ** 22
            for trial in range(20):
                ext = trial < 4                                    # extreme residues first
                u, v = ([[(p - 1) // 2 * (1 if (trial ^ which) & 1 else -1) if ext else
                          rng.randrange(-((p - 1) // 2), (p - 1) // 2 + 1) for _ in range(7)] for p in mods]
                        for which in (0, 1))
                true = [outputs(a, b) for a, b in zip(u, v)]

                tt = [contractands([x + 128 for x in a], [x + 128 for x in b], half) for a, b in zip(u, v)]
                assert all(abs(x) <= 2048 for row in tt for x in row)
                pairs = [[sum(row[e] * (dl[2 * i] + 256 * dl[2 * i + 1]) for row, dl in zip(tt, digits))
                          for i in range(8)] for e in range(4)]
                z = [[a + b for a, b in zip(pairs[0], pairs[1])], [b - a for a, b in zip(pairs[0], pairs[1])],
                     [a - b for a, b in zip(pairs[2], pairs[3])], [-(a + b) for a, b in zip(pairs[2], pairs[3])]]
                for slot in range(4):
                    if half and slot & 1:
                        z[slot] = [-x for x in z[slot]]
                    assert all(abs(x) < 2 ** 31 for x in z[slot])
                    off = nm * 16 * 120 * P - weights[half][slot] * sum(elements)
                    S = off + sum(x << (16 * i) for i, x in enumerate(z[slot]))
                    comp = (4 * half + slot) ^ ((slot & 1) << 2)
                    assert S == nm * 16 * 120 * P + sum(t[comp] * e for t, e in zip(true, elements))


# ------------------------------------------------------------------ GPU
@pytest.fixture(scope="module")
def handles():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with hm.Handle() as default, hm.Handle() as gauss:
        gauss.set_complex_form("gauss")
        yield default, gauss
        assert default.device_error() == 0 and gauss.device_error() == 0


def stored(op, rows, cols):
    return (cols, rows) if op in ("T", "H") else (rows, cols)


# edges of the encoder's 16 x 32 tiles and the 64-deep k-blocks, of the GEMM's 128-row tiles, its output widths and its
# 1024-deep chunks, of the CRT's 32- and 128-column blocks (n = 1024) and of the modulus counts (k = 290 / 291 at 1e-12)
SHAPES = [(1, 1, 1), (16, 32, 64), (17, 33, 65), (128, 256, 290), (129, 257, 291), (40, 1023, 512), (35, 1024, 513),
          (33, 1025, 1024), (130, 70, 1025), (5, 300, 2049)]
OPS = ["N", "T", "C", "H", "QC"]


@pytest.mark.gpu
@pytest.mark.parametrize("tol", [1e-3, 1e-9, 1e-12, 1e-13, 1e-14])
@pytest.mark.parametrize("i", range(len(SHAPES)))
def test_default_form_gives_gausss_bits(handles, i, tol):
    """Both forms recover the same integers and round them once: equal bits, over the digit counts (bits <= 46 and
    above), the limb counts (15 moduli and more), every op, strided operands, complex alpha / beta and plain stores."""
    m, n, k = SHAPES[i]
    opA, opB = OPS[i % 5], OPS[(i * 2 + 1) % 5]
    dev = torch.device("cuda")
    (ra, ca), (rb, cb) = stored(opA, m, k), stored(opB, k, n)
    A = bi.fock_like(800 + i, ra, ca + 3, row_scale=True).to(dev)[:, :, :ca]
    B = bi.uniform(820 + i, rb, cb + 2).to(dev)[:, :, 1:cb + 1]
    C0 = bi.uniform(840 + i, m, n + 5).to(dev)
    for alpha, beta in ((1.0, 0.0), (0.5 - 2j, 0.25 + 1j)):
        outs = []
        for h in handles:
            C = C0.clone()
            hm.hmat_bq_gemm(h, A, B, C[:, :, :n], opA, opB, alpha=alpha, beta=beta, mode="split", tol=tol)
            outs.append(C)
        torch.cuda.synchronize()
        assert torch.equal(outs[0], outs[1])
        assert torch.equal(outs[0][:, :, n:], C0[:, :, n:])


@pytest.mark.gpu
@pytest.mark.parametrize("i", [0, 2, 4, 6, 8])
@pytest.mark.parametrize("fa,fb", [(bi.TRS, bi.TRS), (bi.TRS, bi.TRA), (bi.TRA, bi.TRA), (bi.TRS, bi.BQ),
                                   (bi.BQ, bi.TRA), (bi.TRA, bi.BQ), (bi.COMPLEX, bi.BQ), (bi.BQ, bi.COMPLEX),
                                   (bi.COMPLEX, bi.COMPLEX)])
def test_subalgebra_products_give_gausss_bits(handles, i, fa, fb):
    """The matrix form of each pair of subalgebras it serves, absent components holding NaN; small integers (whose
    exact zeros keep their sign) and wide-ranging data."""
    m, n, k = SHAPES[i]
    opA, opB = OPS[(i + 3) % 5], OPS[i % 5]
    dev = torch.device("cuda")
    (ra, ca), (rb, cb) = stored(opA, m, k), stored(opB, k, n)
    for A, B in ((bi.fock_like(880 + i, ra, ca, row_scale=True), bi.uniform(890 + i, rb, cb)),
                 (bi.small_int(880 + i, ra, ca, lo=-1, hi=1), bi.small_int(890 + i, rb, cb, lo=-1, hi=1))):
        for X, f in ((A, fa), (B, fb)):
            for c in range(8):
                if not (f >> c) & 1:
                    X[c] = float("nan")
        A, B = A.to(dev), B.to(dev)
        C0 = bi.uniform(840 + i, m, n).to(dev)
        for alpha, beta, tol in ((1.0, 0.0, TOL), (0.5 - 2j, 0.25 + 1j, 1e-14)):
            outs = []
            for h in handles:
                C = C0.clone()
                hm.hmat_bq_gemm(h, A, B, C, opA, opB, fa, fb, alpha, beta, mode="split", tol=tol)
                outs.append(C)
            torch.cuda.synchronize()
            assert torch.equal(outs[0].view(torch.int64), outs[1].view(torch.int64))


@pytest.mark.gpu
@pytest.mark.parametrize("use_graph", [False, True])
def test_grouped_matrix_form_beside_other_forms(handles, use_graph):
    """One grouped call of full products (matrix form; k = 5 at tol 1e-3 keeps its plan's form, which then needs fewer
    planes) and subalgebra products: the bits of an all-Gauss handle."""
    dev = torch.device("cuda")
    shapes = [(64, 64, 5, bi.BQ), (130, 70, 64, bi.BQ), (100, 90, 300, bi.TRS), (33, 1030, 200, bi.BQ),
              (50, 60, 70, bi.REAL), (20, 200, 90, bi.COMPLEX), (7, 9, 12, bi.BQ)]
    mats = [(bi.uniform(860 + i, m, k, flags=f).to(dev), bi.uniform(870 + i, k, n).to(dev), f)
            for i, (m, n, k, f) in enumerate(shapes)]
    for tol in (1e-3, TOL):
        res = []
        for h in handles:
            Cs = [torch.full((8, m, n), float("nan"), dtype=torch.float64, device=dev) for m, n, _, _ in shapes]
            descs = [hm.make_desc(A, B, C, flagsA=f) for (A, B, f), C in zip(mats, Cs)]
            ws = torch.empty(hm.hmat_workspace_size(h, descs, "split", tol), dtype=torch.uint8, device=dev)
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            for _ in range(2 if use_graph else 1):
                hm.hmat_bq_gemm_grouped(h, descs, mode="split", tol=tol, workspace=ws, stream=s, use_graph=use_graph)
            s.synchronize()
            res.append(Cs)
        for a, b in zip(*res):
            assert torch.equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("fa,fb", [(bi.BQ, bi.BQ), (bi.TRS, bi.BQ), (bi.TRS, bi.TRA), (bi.COMPLEX, bi.BQ)])
@pytest.mark.parametrize("m,n", [(5, 9), (130, 70), (300, 257)])
def test_half_last_k_block(m, n, fa, fb):
    """The last 64-deep k-block is kept as a half block when it holds at most 32 of k: exact on small
    integers on both sides of every boundary, and of the accumulation chunks (up to 1088 deep, spread evenly)."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with hm.Handle() as h:
        for k in (1, 16, 31, 32, 33, 63, 64, 65, 80, 96, 97, 128, 150, 1024, 1025, 1057, 1088, 1089, 2090, 2177):
            A, B = bi.small_int(800 + k, m, k, flags=fa), bi.small_int(801 + k, k, n, flags=fb)
            want = torch.full((8, m, n), float("nan"), dtype=torch.float64, device="cuda")
            got = want.clone()
            Ad, Bd = A.cuda(), B.cuda()
            hm.hmat_bq_gemm(h, Ad, Bd, want, flagsA=fa, flagsB=fb, mode="fp64")      # exact on small integers
            hm.hmat_bq_gemm(h, Ad, Bd, got, flagsA=fa, flagsB=fb, mode="split", tol=TOL)
            assert torch.equal(got, want), k
        assert h.device_error() == 0


@pytest.mark.gpu
def test_narrow_products_beside_deep_ones():
    """Products of one accumulation chunk in a launch with deeper ones, over output widths whose halves
    the epilogue splits unevenly (32: one half only; 96, 160, 224): exact on small integers."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    shapes = [(40, 20, 100), (70, 33, 1500), (10, 32, 64), (140, 32, 1300), (200, 224, 2100), (33, 90, 700), (150, 160, 1090),
              (129, 100, 3000)]
    with hm.Handle() as h:
        descs, outs = [], []
        for i, (m, n, k) in enumerate(shapes):
            A, B = bi.small_int(830 + i, m, k).cuda(), bi.small_int(840 + i, k, n).cuda()
            C, want = (torch.full((8, m, n), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
            hm.hmat_bq_gemm(h, A, B, want, mode="fp64")
            descs.append(hm.make_desc(A, B, C))
            outs.append((C, want, A, B))
        hm.hmat_bq_gemm_grouped(h, descs, "split", TOL)
        for i, (C, want, _, _) in enumerate(outs):
            assert torch.equal(C, want), shapes[i]
            C.fill_(float("nan"))
        for d, (C, want, A, B) in zip(descs, outs):
            hm.hmat_bq_gemm(h, A, B, C, mode="split", tol=TOL)
            assert torch.equal(C, want)
        assert h.device_error() == 0


def test_running_sums_of_chunk_residues():
    """The GEMM's accumulation chunks: 1088-deep sums of products of the matrix form's residues (up to 121) are exact in
    FP32, and so are the running sums of the chunks' residues (up to 129), 254 of them at the largest k in the
    four-multiplication form, whose depth is 2 k."""
    assert 1088 * 121 ** 2 < 2 ** 24
    kmax = max(k for k in (127 * 1024, 127 * 1024 + 1) if _served(k))
    assert kmax == 127 * 1024
    assert 129 * (2 * kmax // 1024) < 2 ** 15


def _served(k):
    try:
        hm.split_info(k, TOL)
    except hm.HmatError:
        return False
    return True
