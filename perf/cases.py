"""The workloads by which this library's speed is followed.

A case is one call (or one short sequence of calls) that a user's program
makes through the public entry points: single products in both modes, grouped
products, products streamed from host memory and the data movement around a
diagonalisation.  Sizes are those of the repository's benchmark configurations
(n = 256, 4096 and 8192, the batch of 512 products with dimensions
log-uniform in [32, 1024]) and ragged ones in between.

Matrices are (8, rows, cols) float64 tensors of the components [M1..M8];
the complex coefficient of basis element e is M_e + i M_{e+4}.
"""
import math
import random

import torch

import paper_2609_02081_gb300 as hm

BQ, TRS, TRA, COMPLEX = 0xFF, 0x0F, 0xF0, 0x11

# signs of the stored components under each op (T and H also transpose)
_SIGNS = {"N": (1, 1, 1, 1, 1, 1, 1, 1), "T": (1, 1, -1, 1, 1, 1, -1, 1), "C": (1, -1, 1, -1, -1, 1, -1, 1),
          "H": (1, -1, -1, -1, -1, 1, 1, 1), "QC": (1, -1, -1, -1, 1, -1, -1, -1)}

_the_handle = None


def _handle():
    """The one handle a program creates at start-up."""
    global _the_handle
    if _the_handle is None:
        _the_handle = hm.Handle()
    return _the_handle


def _gemm(name, m, n, k, mode, opA="N", opB="N", fa=BQ, fb=BQ, alpha=(1.0, 0.0), beta=(0.0, 0.0), tol=1e-12,
          data="fock"):
    return {"name": name, "kind": "gemm", "m": m, "n": n, "k": k, "mode": mode, "opA": opA, "opB": opB, "fa": fa,
            "fb": fb, "ar": alpha[0], "ai": alpha[1], "br": beta[0], "bi": beta[1], "tol": tol, "data": data}


def listed():
    return [
        # the smallest benchmark configuration: one small product, where launches and latency count
        _gemm("split-n256", 256, 256, 256, "split"),
        # a Fock-sized product with the Hermitian conjugate of the left operand (similarity transforms)
        _gemm("split-n4096-H", 4096, 4096, 4096, "split", opA="H"),
        # time-reversal symmetric times antisymmetric: the real-quaternion subalgebras
        _gemm("split-n4096-trs-tra", 4096, 4096, 4096, "split", fa=TRS, fb=TRA),
        # the headline: a Fock-like matrix with rows of very different scale
        _gemm("split-n8192-fock", 8192, 8192, 8192, "split", data="fock_rows"),
        # a block of a larger matrix: odd sizes, transposed and conjugated operands, complex scalars, update of C
        _gemm("split-ragged-update", 1537, 771, 2049, "split", opA="T", opB="C", alpha=(0.5, -1.25),
              beta=(0.25, 0.5), data="uniform"),
        # a complex matrix (a spin-free orbital basis) applied to a full one
        _gemm("split-complex-bq", 3000, 1000, 2000, "split", fa=COMPLEX, data="uniform"),
        # the batch configuration: 512 products of very different shapes in one call
        {"name": "grouped-512", "kind": "grouped", "count": 512, "lo": 32, "hi": 1024, "shapes": 104},
        # a batch of small blocks (one molecule's shells)
        {"name": "grouped-64-small", "kind": "grouped", "count": 64, "lo": 32, "hi": 160, "shapes": 7},
        # plain FP64 mode, for callers who want FP64 rounding: small and large
        _gemm("fp64-n256", 256, 256, 256, "fp64", data="uniform"),
        _gemm("fp64-n2048", 2048, 2048, 2048, "fp64"),
        # operands and result in pinned host memory, computed within a device budget
        {"name": "streamed-n3072", "kind": "streamed", "m": 3072, "n": 3072, "k": 3072, "budget_gb": 16},
        # before and after an eigensolver: Hermitian part, check, complex image and back
        {"name": "hermitian-n4096", "kind": "hermitian", "n": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["split", "split", "split", "split", "grouped", "fp64", "streamed", "hermitian"])
    if kind in ("split", "fp64"):
        hi = 4096 if kind == "split" else 1024
        m, n, k = (_log_int(rng, 32, hi) for _ in range(3))
        fa, fb = rng.choice([(BQ, BQ), (BQ, BQ), (BQ, BQ), (TRS, TRA), (TRS, BQ), (COMPLEX, BQ), (BQ, COMPLEX)])
        scalars = rng.choice([((1.0, 0.0), (0.0, 0.0)), ((1.0, 0.0), (0.0, 0.0)), ((0.75, -0.5), (0.5, 0.25))])
        c = _gemm("", m, n, k, kind, rng.choice(list(_SIGNS)), rng.choice(list(_SIGNS)), fa, fb, scalars[0],
                  scalars[1], rng.choice([1e-12, 1e-12, 1e-9, 1e-14]), rng.choice(["fock", "fock_rows", "uniform"]))
        del c["name"]
        return c
    if kind == "grouped":
        return {"kind": "grouped", "count": _log_int(rng, 4, 256), "lo": 32, "hi": _log_int(rng, 64, 1024),
                "shapes": rng.randrange(1 << 20)}
    if kind == "streamed":
        m, n, k = (_log_int(rng, 512, 3072) for _ in range(3))
        return {"kind": "streamed", "m": m, "n": n, "k": k, "budget_gb": rng.choice([4, 8, 16])}
    return {"kind": "hermitian", "n": _log_int(rng, 64, 4096)}


# ------------------------------------------------------------------ inputs
def _fill(X, gen, flags, data):
    """Random entries in the present components of X (8, rows, cols), zeros in the others."""
    rows, cols = X.shape[1], X.shape[2]
    if data == "uniform":
        X.copy_(torch.rand(X.shape, generator=gen, device=X.device, dtype=torch.float64).mul_(2.0).sub_(1.0))
    else:                                        # banded, decaying away from the diagonal
        X.copy_(torch.randn(X.shape, generator=gen, device=X.device, dtype=torch.float64))
        i = torch.arange(rows, device=X.device, dtype=torch.float64).view(rows, 1)
        j = torch.arange(cols, device=X.device, dtype=torch.float64).view(1, cols)
        X.mul_(torch.exp((i - j).abs_().mul_(-1.0 / 200.0)))
        if data == "fock_rows":                  # row scales 10**U(-6, 0)
            u = torch.rand((rows, 1), generator=gen, device=X.device, dtype=torch.float64)
            X.mul_(torch.pow(10.0, -6.0 * u))
    for c in range(8):
        if not (flags >> c) & 1:
            X[c].zero_()
    return X


def _random(gen, rows, cols, flags, data):
    return _fill(torch.empty((8, rows, cols), dtype=torch.float64, device="cuda"), gen, flags, data)


def _stored(op, rows, cols):
    return (cols, rows) if op in ("T", "H") else (rows, cols)


def _batch_shapes(case):
    r = random.Random(case["shapes"])
    return [tuple(_log_int(r, case["lo"], case["hi"]) for _ in range(3)) for _ in range(case["count"])]


def _batch_views(case, which):
    """Total doubles and (offset, rows, cols) of each problem's A (0), B (1) or C (2) in one flat buffer."""
    at, out = 0, []
    for m, n, k in _batch_shapes(case):
        rows, cols = ((m, k), (k, n), (m, n))[which]
        out.append((at, rows, cols))
        at += (8 * rows * cols + 31) // 32 * 32
    return at, out


def _views(flat, layout):
    return [flat[at:at + 8 * r * c].view(8, r, c) for at, r, c in layout]


def _inputs(case, seed):
    """The operands alone, in device memory (streamed operands are copied to the host by prepare)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return (_random(gen, *_stored(case["opA"], m, k), case["fa"], case["data"]),
                _random(gen, *_stored(case["opB"], k, n), case["fb"], case["data"]),
                _random(gen, m, n, BQ, "uniform") if (case["br"], case["bi"]) != (0.0, 0.0) else
                torch.zeros((8, m, n), dtype=torch.float64, device="cuda"))
    if kind == "grouped":
        return tuple(torch.rand(_batch_views(case, w)[0], generator=gen, device="cuda",
                                dtype=torch.float64).mul_(2.0).sub_(1.0) for w in (0, 1))
    if kind == "streamed":
        m, n, k = case["m"], case["n"], case["k"]
        return _random(gen, m, k, BQ, "fock"), _random(gen, k, n, BQ, "fock")
    n = case["n"]
    return (_random(gen, n, n, BQ, "fock"),)


def prepare(case, seed):
    h = _handle()
    kind = case["kind"]
    x = _inputs(case, seed)
    s = {"case": case, "h": h}
    if kind == "gemm":
        s["A"], s["B"], s["C"] = x
        d = hm.make_desc(*x, case["opA"], case["opB"], case["fa"], case["fb"], complex(case["ar"], case["ai"]),
                         complex(case["br"], case["bi"]))
        nbytes = hm.hmat_workspace_size(h, [d], case["mode"], case["tol"])
        # a program keeps its workspace, unless it is so large that it is taken from the allocator for the call
        s["ws"] = torch.empty(max(nbytes, 1), dtype=torch.uint8, device="cuda") if nbytes < (40 << 30) else None
    elif kind == "grouped":
        C = torch.zeros(_batch_views(case, 2)[0], dtype=torch.float64, device="cuda")
        s["flat"] = (x[0], x[1], C)
        s["descs"] = [hm.make_desc(a, b, c) for a, b, c in
                      zip(*(_views(f, _batch_views(case, w)[1]) for w, f in enumerate(s["flat"])))]
        s["ws"] = torch.empty(hm.hmat_workspace_size(h, s["descs"], "split", 1e-12), dtype=torch.uint8, device="cuda")
    elif kind == "streamed":
        s["A"], s["B"] = (torch.empty(t.shape, dtype=torch.float64, pin_memory=True).copy_(t) for t in x)
        s["C"] = torch.zeros((8, case["m"], case["n"]), dtype=torch.float64).pin_memory()
        s["ws"] = torch.empty(case["budget_gb"] << 30, dtype=torch.uint8, device="cuda")
    else:
        n = case["n"]
        s["F"] = x[0]
        s["H"] = torch.empty_like(x[0])
        s["Y"] = torch.empty_like(x[0])
        s["Z"] = torch.empty((2 * n, 2 * n), dtype=torch.complex128, device="cuda")
    return s


def run(s):
    case, h = s["case"], s["h"]
    kind = case["kind"]
    if kind == "gemm":
        return hm.hmat_bq_gemm(h, s["A"], s["B"], s["C"], case["opA"], case["opB"], case["fa"], case["fb"],
                               complex(case["ar"], case["ai"]), complex(case["br"], case["bi"]), mode=case["mode"],
                               tol=case["tol"], workspace=s["ws"])
    if kind == "grouped":
        hm.hmat_bq_gemm_grouped(h, s["descs"], mode="split", tol=1e-12, workspace=s["ws"])
        return s["flat"][2]
    if kind == "streamed":
        return hm.hmat_bq_gemm_streamed(h, s["A"], s["B"], s["C"], mode="split", tol=1e-12, workspace=s["ws"])
    hm.hmat_bq_add(h, s["F"], s["F"], s["H"], alpha=0.5, beta=0.5, opB="H")
    off = hm.hmat_bq_hermiticity(h, s["H"])
    hm.hmat_bq_to_complex(h, s["H"], s["Z"])
    hm.hmat_complex_to_bq(h, s["Z"], s["Y"])
    return s["H"], off, s["Z"], s["Y"]


# ------------------------------------------------------------------ what a pass cannot do without
def _popcount(flags):
    return bin(flags).count("1")


def _products(fa, fb):
    """Real matrix products of the bilinear scheme for these component flags."""
    return {(BQ, BQ): 24, (TRS, TRA): 8, (TRS, BQ): 16, (COMPLEX, BQ): 12, (BQ, COMPLEX): 12}[(fa, fb)]


def work(case):
    kind = case["kind"]
    if kind in ("gemm", "streamed"):
        m, n, k = case["m"], case["n"], case["k"]
        fa, fb = case.get("fa", BQ), case.get("fb", BQ)
        update = (case.get("br", 0.0), case.get("bi", 0.0)) != (0.0, 0.0)
        return {"bytes": 8 * (_popcount(fa) * m * k + _popcount(fb) * k * n + 8 * m * n * (2 if update else 1)),
                "flops": 2 * _products(fa, fb) * m * n * k}
    if kind == "grouped":
        shapes = _batch_shapes(case)
        return {"bytes": sum(64 * (m * k + k * n + m * n) for m, n, k in shapes),
                "flops": sum(48 * m * n * k for m, n, k in shapes)}
    n = case["n"]
    return {"bytes": 64 * n * n * 4, "flops": 16 * n * n}


# ------------------------------------------------------------------ the same in plain 64-bit torch
def _image(X, op="N"):
    """The complex 2 rows x 2 cols image of op(X): [[q1 + i q2, q3 + i q4], [-q3 + i q4, q1 - i q2]]."""
    M = [X[c] * float(_SIGNS[op][c]) for c in range(8)]
    if op in ("T", "H"):
        M = [c.transpose(0, 1) for c in M]
    q = [torch.complex(M[e].contiguous(), M[e + 4].contiguous()) for e in range(4)]
    return torch.cat([torch.cat([q[0] + 1j * q[1], q[2] + 1j * q[3]], 1),
                      torch.cat([-q[2] + 1j * q[3], q[0] - 1j * q[1]], 1)], 0)


def _components(Z):
    """The eight components of a complex 2 rows x 2 cols image of that kind."""
    m, n = Z.shape[0] // 2, Z.shape[1] // 2
    a, b, c, d = Z[:m, :n], Z[:m, n:], Z[m:, :n], Z[m:, n:]
    q = [(a + d) * 0.5, (a - d) * -0.5j, (b - c) * 0.5, (b + c) * -0.5j]
    return torch.stack([x.real for x in q] + [x.imag for x in q])


def _product(A, B, opA="N", opB="N"):
    return _components(_image(A, opA) @ _image(B, opB))


def _scale(X, z):
    re, im = X[:4], X[4:]
    return torch.cat([re * z.real - im * z.imag, re * z.imag + im * z.real])


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        if case["m"] * case["n"] * case["k"] > 1 << 37:
            return None                          # a plain FP64 product of that size takes most of a minute
        A, B, C = _inputs(case, seed)
        P = _scale(_product(A, B, case["opA"], case["opB"]), complex(case["ar"], case["ai"]))
        return P + _scale(C, complex(case["br"], case["bi"]))
    if kind == "grouped":
        flat = _inputs(case, seed)
        C = torch.zeros(_batch_views(case, 2)[0], dtype=torch.float64, device="cuda")
        for a, b, c in zip(*(_views(f, _batch_views(case, w)[1]) for w, f in enumerate((*flat, C)))):
            c.copy_(_product(a, b))
        return C
    if kind == "streamed":
        return _product(*_inputs(case, seed)).cpu()
    F, = _inputs(case, seed)
    sign = torch.tensor(_SIGNS["H"], dtype=torch.float64, device="cuda").view(8, 1, 1)
    H = 0.5 * F + 0.5 * (F.transpose(1, 2) * sign)
    off = (H - H.transpose(1, 2) * sign).abs().max().view(1)
    # the library's complex image is taken in another basis; its inverse gives H back
    E, Fq, G, K = (torch.complex(H[0], H[1]), torch.complex(H[2], H[3]), torch.complex(-H[5], H[4]),
                   torch.complex(-H[7], H[6]))
    Z = torch.cat([torch.cat([E + G, Fq + K], 1), torch.cat([-Fq.conj() + K.conj(), E.conj() - G.conj()], 1)], 0)
    return H, off, Z, H
