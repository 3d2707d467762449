"""The sweep's 32 x 32 cells at the sizes where they can go wrong: edges of leaves (8), cells (32) and tiles (128), odd leading dimensions,
matrices of a batch that are swept by themselves, and values that look like the mark of an entry that has not arrived."""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import cref
from certify import certified_case
from paper_2607_27042_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_2607_27042_b200 import gptq2d
    return gptq2d


def padded(a, extra):
    r, c = a.shape
    buf = torch.full((r, c + extra), float("nan"), dtype=torch.float64, device="cuda")
    buf[:, :c] = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return buf[:, :c]


def certified(m, n, seed):
    def draw(s):
        X, A, B = W.gaussian_like(m, n, s)
        L, U, _, _ = O.feedback_factors(A, B)
        return X, L, U
    return certified_case(draw, cref.nested, seed)[:2]


@pytest.mark.parametrize("m,n,extra", [(7, 8, 0), (8, 33, 1), (31, 32, 0), (33, 31, 1), (32, 64, 2), (63, 97, 1), (96, 128, 0), (65, 129, 3),
                                       (128, 160, 1), (161, 95, 0), (127, 393, 1), (421, 225, 0)])
def test_edges_of_leaves_cells_and_tiles(g, m, n, extra):
    (X, L, U), ref = certified(m, n, 10 * m + n)
    Z, E, mm, info = g.gptq2d_round(padded(X, extra), padded(L, extra), padded(U, extra), want_E=True, want_margin=True)
    g.check_info(info)
    assert np.array_equal(Z.cpu().numpy().astype(np.int64), ref["Z"])
    # sums of at most 800 fp64 terms of order one in two orders: the bar of all error comparisons in these tests
    assert np.max(np.abs(E.cpu().numpy() - ref["E"])) < 1e-9 and abs(float(mm[0]) - ref["margin"]) < 1e-9


def test_matrices_of_a_batch_swept_by_themselves(g):
    shapes = [(100, 130), (64, 64), (300, 140), (33, 40), (129, 260)]      # 16, 16, 48, 16 and 48 cells, tiles counted whole
    cases = [certified(m, n, 77 + k) for k, (m, n) in enumerate(shapes)]
    args = [[padded(c[0][q], 0) for c in cases] for q in range(3)]
    whole = g.gptq2d_round_batched(*args, want_E=True, want_margin=True)
    g.gptq2d_internal_test_hook(8, 5)                                      # cell indices of 5 bits: two matrices do not fit
    try:
        parts = g.gptq2d_round_batched(*args, want_E=True, want_margin=True)
    finally:
        g.gptq2d_internal_test_hook(8, 0)
    for info in (whole[3], parts[3]):
        g.check_info(info)
    for b, (_, ref) in enumerate(cases):
        assert np.array_equal(parts[0][b].cpu().numpy().astype(np.int64), ref["Z"])
        assert torch.equal(parts[0][b], whole[0][b]) and torch.equal(parts[1][b], whole[1][b])
    assert torch.equal(parts[2], whole[2])


@pytest.mark.parametrize("i,j", [(0, 0), (40, 70), (150, 20)])
def test_a_nan_that_looks_like_a_missing_entry_is_an_ordinary_nan(g, i, j):
    mark = 0xfff94d5a7c3e2b61
    X, A, B = W.gaussian_like(160, 170, 5)
    L, U, _, _ = O.feedback_factors(A, B)
    X[i, j] = np.array([mark], dtype=np.uint64).view(np.float64)[0]
    ws = torch.zeros(g.gptq2d_round_workspace_bytes(160, 170) // 8, dtype=torch.int64, device="cuda")
    Z, E, mm, info = g.gptq2d_round(padded(X, 0), padded(L, 0), padded(U, 0), want_E=True, workspace=ws.view(torch.uint8))
    vals = info.cpu().tolist()
    assert vals[0] == 6 and abs(vals[1] + vals[2] - i - j) < 15            # known to a leaf's 15 anti-diagonals
    # the caller's E is stored as computed: entries with the mark's bits did come up; none of them was posted with these bits
    assert (E.cpu().numpy().view(np.uint64) == mark).any()
    posted = ws.cpu().numpy().view(np.uint64)
    assert not (posted == mark).any() and (posted == mark ^ 1).any()
