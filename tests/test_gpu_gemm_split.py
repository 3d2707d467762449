"""The fp64 product on the int8 tensor cores (error-free splitting into base-256 digits) against exact integers and
against a bound on what its digits drop."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_2607_27042_b200 import gptq2d
    return gptq2d


def padded(a):
    r, c = a.shape
    buf = torch.full((r, c + 3), 7.0, dtype=torch.float64, device="cuda")     # odd pitches among them
    buf[:, :c] = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return buf[:, :c]


@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (1, 1, 1), (127, 129, 65), (257, 130, 191), (300, 100, 1000),
                                   (129, 2200, 128), (8, 513, 4100)])
def test_integers_are_exact_in_all_layouts(g, M, N, K):
    rng = np.random.default_rng(M * 1000003 + N * 1009 + K)
    for transa in (False, True):
        for transb in (False, True):
            a = rng.integers(-8, 9, size=(M, K)).astype(np.float64)
            b = rng.integers(-8, 9, size=(K, N)).astype(np.float64)
            c0 = rng.integers(-8, 9, size=(M, N)).astype(np.float64)
            for beta in (-1.0, 0.0):
                c = padded(c0)
                info = torch.full((4,), 9, dtype=torch.int32, device="cuda")
                g.gptq2d_internal_gemm_split(padded(a.T if transa else a), padded(b.T if transb else b), c, transa=transa,
                                             transb=transb, alpha=2.0, beta=beta, info=info)
                g.check_info(info)
                assert np.array_equal(c.cpu().numpy(), 2.0 * (a @ b) + beta * c0), (transa, transb, beta)


@pytest.mark.parametrize("K", [1, 100, 1024])
def test_rounding_is_within_the_digits_that_are_kept(g, K):
    # rows over 200 binary orders, entries of a row over 12; a row of zeros, a tiny one, one with a single entry at the
    # top of its binade
    rng = np.random.default_rng(K)
    M, N = 150, 200
    a = rng.standard_normal((M, K)) * np.exp2(rng.integers(-100, 100, size=(M, 1))) * np.exp2(rng.integers(-12, 1, size=(M, K)))
    b = rng.standard_normal((K, N)) * np.exp2(rng.integers(-100, 100, size=(1, N)))
    a[3] = 0.0
    a[4] *= 1e-200
    a[5, 0] = np.nextafter(2.0, 0.0) * 2.0 ** 60
    c = torch.empty((M, N), dtype=torch.float64, device="cuda")
    g.gptq2d_internal_gemm_split(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), c)
    want = a.astype(np.longdouble) @ b.astype(np.longdouble)
    # digits: half a unit of 2^-56 on either side, five dropped pairs of weight 256^-10 and fewer beyond; a scale is at most
    # 4.04 times the largest entry: K * 16.4 * (2^-57 + 2^-64) < K * 2^-52.9; then the rounding of the result
    top = np.abs(a).max(1, initial=0.0)[:, None] * np.abs(b).max(0, initial=0.0)[None, :]
    bound = K * 2.0 ** -52.9 * top + 2.0 ** -51 * np.abs(want).astype(np.float64)
    assert np.all(np.abs(c.cpu().numpy() - want) <= bound)


def test_non_finite_entries_reach_their_row_and_column_only(g):
    rng = np.random.default_rng(1)
    a, b = rng.standard_normal((140, 70)), rng.standard_normal((70, 150))
    clean = a @ b
    a[7, 3], b[5, 139] = np.nan, np.inf
    c = torch.empty((140, 150), dtype=torch.float64, device="cuda")
    g.gptq2d_internal_gemm_split(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), c)
    c = c.cpu().numpy()
    assert np.all(~np.isfinite(c[7])) and np.all(~np.isfinite(c[:, 139]))
    c[7], c[:, 139], clean[7], clean[:, 139] = 0, 0, 0, 0
    assert np.max(np.abs(c - clean)) < 1e-13
