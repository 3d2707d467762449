"""Resident sweeps in 2 x 2 blocks (the route of large matrices) at small sizes: blocks of one tile and of several, ragged last tiles, odd
leading dimensions, products whose residue planes fit only piece by piece."""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import cref
from certify import certified_case
from paper_2607_27042_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture()
def g():
    from paper_2607_27042_b200 import gptq2d
    gptq2d.gptq2d_internal_test_hook(7, 129)
    yield gptq2d
    gptq2d.gptq2d_internal_test_hook(7, 0)


def padded(a, extra):
    r, c = a.shape
    buf = torch.full((r, c + extra), float("nan"), dtype=torch.float64, device="cuda")
    buf[:, :c] = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return buf[:, :c]


def workspace(g, m, n, room):
    """Room for everything, for all but the residue planes, or for the bookkeeping alone: what is missing lies in free rows."""
    size = g.gptq2d_round_workspace_bytes(m, n)
    m0, n0 = ((-(-k // 128) + 1) // 2 * 128 for k in (m, n))
    if room != "all":
        size -= 16 * (m0 + n0) * max(m0, n0)
    if room == "none":                                   # scales, tops and bits of an operand's rows, scaling along k
        up = lambda x: -(-x // 256) * 256
        size -= sum(up(8 * k) + up(12 * k + k // 16) for k in (m0, n0)) + up(8 * max(m0, n0))
    return torch.full((size,), 0xff, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("room", ["planes missing", "none"])
@pytest.mark.parametrize("m,n,extra", [(780, 900, 1), (769, 1900, 3), (1500, 800, 1), (1027, 1290, 0)])
def test_planes_in_free_rows(g, m, n, extra, room):
    # k in two pieces and more; ragged last tiles, odd pitches, an outlier channel of integers.  The same sums as with room for the planes, in
    # more pieces: a rounding of the result a piece.
    X, A, B = W.gaussian_like(m, n, m + n)
    L, U, _, _ = O.feedback_factors(A, B)
    X[0] = np.round(X[0])
    L[1:, 0] *= 1e6
    dX, dL, dU = padded(X, extra), padded(L, extra), padded(U, extra)
    out = []
    for r in ("all", room):
        ws = workspace(g, m, n, r)
        out.append(g.gptq2d_round(dX, dL, dU, workspace=ws, want_E=True, want_margin=True) + (g.gptq2d_internal_round_products(m, n, ws.numel()),))
        g.check_info(out[-1][3])
    (Z0, E0, mm0, _, n0), (Z1, E1, mm1, _, n1) = out
    assert n0 == 4 and n1 > 4, n1
    assert torch.equal(Z0, Z1) and float((E0 - E1).abs().max()) < 1e-13 and abs(float(mm0[0]) - float(mm1[0])) < 1e-13
    g.gptq2d_internal_test_hook(7, 0)
    Z2, E2, _, info = g.gptq2d_round(dX, dL, dU, want_E=True)
    g.check_info(info)
    # sums of at most 2900 terms of order one in fp64
    assert torch.equal(Z2, Z1) and float((E2 - E1).abs().max()) < 1e-12


@pytest.mark.parametrize("m,n,extra", [(129, 130, 0), (256, 256, 0), (300, 330, 1), (200, 1000, 2), (1000, 140, 3), (770, 645, 0)])
def test_blocks_equal_the_oracle_and_the_single_sweep(g, m, n, extra):
    def draw(seed):
        X, A, B = W.gaussian_like(m, n, seed)
        L, U, _, _ = O.feedback_factors(A, B)
        return X, L, U
    (X, L, U), ref, _ = certified_case(draw, cref.nested, m + n)
    dX, dL, dU = padded(X, extra), padded(L, extra), padded(U, extra)
    ws = torch.full((g.gptq2d_round_workspace_bytes(m, n),), 0xff, dtype=torch.uint8, device="cuda")
    Z, E, mm, info = g.gptq2d_round(dX, dL, dU, workspace=ws, want_E=True, want_margin=True)
    g.check_info(info)
    assert np.array_equal(Z.cpu().numpy().astype(np.int64), ref["Z"])
    g.gptq2d_internal_test_hook(7, 0)
    Z1, E1, mm1, info = g.gptq2d_round(dX, dL, dU, want_E=True, want_margin=True)
    g.check_info(info)
    assert torch.equal(Z, Z1)
    # both sum the same terms in fp64: the bar of all error comparisons in these tests
    assert float((E - E1).abs().max()) < 1e-9 and abs(float(mm[0]) - float(mm1[0])) < 1e-9


@pytest.mark.parametrize("where", [[(7, 20)], [(400, 30)], [(20, 500)], [(380, 470)], [(250, 250), (2, 400)]])
def test_status_words_name_the_first_anti_diagonal(g, where):
    X, A, B = W.gaussian_like(410, 520, 3)
    L, U, _, _ = O.feedback_factors(A, B)
    for i, j in where:
        X[i, j] = np.nan
    Z, E, mm, info = g.gptq2d_round(padded(X, 0), padded(L, 0), padded(U, 0))
    vals = info.cpu().tolist()
    i, j = min(where, key=lambda p: p[0] + p[1])
    # inside an 8 x 8 leaf a NaN reaches entries that exact arithmetic would spare: the anti-diagonal is known to a leaf's 15
    assert vals[0] == 6 and abs(vals[1] + vals[2] - i - j) < 15 and vals[3] == 0


@pytest.mark.parametrize("m,n", [(300, 330), (515, 400)])
def test_an_outlier_channel_of_integers_costs_no_digits(g, m, n):
    # row 0 of X is whole numbers: its errors are zero, and so is what the large entries of column 0 of L are multiplied by
    X, A, B = W.gaussian_like(m, n, 11)
    L, U, _, _ = O.feedback_factors(A, B)
    X[0] = np.round(X[0])
    L[1:, 0] *= 1e6
    dX, dL, dU = padded(X, 0), padded(L, 0), padded(U, 0)
    Z, E, _, info = g.gptq2d_round(dX, dL, dU, want_E=True)
    g.check_info(info)
    g.gptq2d_internal_test_hook(7, 0)
    Z1, E1, _, info = g.gptq2d_round(dX, dL, dU, want_E=True)
    g.check_info(info)
    # sums of at most 900 terms of order one in fp64, each side: 900 * 2^-53
    assert torch.equal(Z, Z1) and float((E - E1).abs().max()) < 1e-13


def error(E, Z, X, L, U):
    """2-norm of the error of E over that of E.  L E U = Z - X whatever the integers are: the residual in 64-bit significands, solved for."""
    w = np.longdouble
    R = (Z.astype(w) - X.astype(w) - (L.astype(w) @ E.astype(w)) @ U.astype(w)).astype(np.float64)
    return np.linalg.norm(np.linalg.solve(L, np.linalg.solve(U.T, R.T).T)) / np.linalg.norm(E)


@pytest.mark.parametrize("room", ["all", "planes missing"])
@pytest.mark.parametrize("kind", ["plain", "scaled", "heavy", "spectrum"])
def test_blocks_lose_no_precision(g, kind, room):
    m, n = 640, 700
    rng = np.random.default_rng(21)
    sigma = {"plain": 0.0, "scaled": 1.0, "heavy": 1.5}

    def basis(k):
        if kind == "spectrum":
            q = np.linalg.qr(rng.standard_normal((k, k)))[0]
            s = (q * np.logspace(0, -6, k)) @ q.T
        else:
            s = rng.standard_normal((k, 2 * k)) * np.exp(sigma[kind] * rng.standard_normal((k, 1)))
            s = s @ s.T / (2 * k)
            s += 0.01 * np.mean(np.diag(s)) * np.eye(k)
        return np.linalg.cholesky(0.5 * (s + s.T)).T.copy()
    L, U, _, _ = O.feedback_factors(basis(m), basis(n))
    X = 4.0 * rng.standard_normal((m, n))
    err = []
    for order in (1 << 30, 129):
        g.gptq2d_internal_test_hook(7, order)
        ws = workspace(g, m, n, room) if order == 129 else None
        Z, E, _, info = g.gptq2d_round(padded(X, 0), padded(L, 0), padded(U, 0), workspace=ws, want_E=True)
        g.check_info(info)
        err.append(error(E.cpu().numpy(), Z.cpu().numpy(), X, L, U))
    # the same sums, half of them rounded once (once a piece of k) instead of once a term
    assert err[1] <= 1.05 * err[0], err
