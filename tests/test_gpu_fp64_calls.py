"""FP64 calls whose tiles leave SMs idle: which cut of the inner dimension they get.

The rounding of a random product tells the cuts apart, so equal bits mean the same cut.
"""
import numpy as np
import pytest
import torch

import bq_inputs as bi
import paper_2609_02081_gb300 as hm

pytestmark = pytest.mark.gpu


@pytest.fixture
def handle():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with hm.Handle() as h:
        yield h
        assert h.device_error() == 0


def grouped(h, probs, ws, use_graph):
    """The grouped FP64 call into the problems' own outputs; returns copies of them."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    hm.hmat_bq_gemm_grouped(h, [hm.make_desc(*p) for p in probs], "fp64", workspace=ws, stream=s, use_graph=use_graph)
    s.synchronize()
    return [c.clone() for _, _, c in probs]


def problem(seed, m, n, k):
    return (bi.uniform(seed, m, k).cuda(), bi.uniform(seed + 1, k, n).cuda(),
            torch.zeros((8, m, n), dtype=torch.float64, device="cuda"))


def test_graph_follows_the_split_k_table(handle):
    """A call replayed from a graph is cut as the table installed when it is made says, like
    the eager call: the rule's ranges, two slices, the ranges again."""
    probs = [problem(900, 64, 64, 512)]
    ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    two = np.full((16, 16), 2, dtype=np.int8)
    seen = []
    for table in (None, two, None):
        handle.set_fp64_splitk_table(table)
        eager = grouped(handle, probs, ws, False)
        for _ in range(2):
            assert torch.equal(grouped(handle, probs, ws, True)[0], eager[0])
        seen.append(eager[0])
    assert torch.equal(seen[0], seen[2]) and not torch.equal(seen[0], seen[1])


@pytest.mark.parametrize("algo", ["bilinear", "isomorph"])
@pytest.mark.parametrize("m0", [32, 200])
def test_reported_workspace_holds_the_cut(handle, algo, m0):
    """Beside a product without an inner dimension (which no algorithm enlarges, and whose plan
    is empty) the reported workspace is what the call's cut needs: more changes nothing."""
    handle.set_algorithm(algo)
    probs = [problem(910, 64, 64, 256), problem(920, m0, m0, 0)]
    need = hm.hmat_workspace_size(handle, [hm.make_desc(*p) for p in probs], "fp64")
    big = torch.empty(need + (64 << 20), dtype=torch.uint8, device="cuda")
    first = grouped(handle, probs, big[:need], False)
    assert torch.equal(grouped(handle, probs, big, False)[0], first[0])
