"""The fp64 product on the int8 tensor cores (residues of 56-bit integers) against exact integers and against a bound on
what its digits drop."""
import numpy as np
import pytest
import torch

import oracle as O

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


@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (5, 3, 2), (127, 129, 65), (257, 130, 191), (300, 100, 1000)])
@pytest.mark.parametrize("why", ["fp64", "scaled along k"])
def test_integers_are_exact_in_all_layouts_where_digits_alone_do_not_do(g, M, N, K, why):
    # "fp64": magnitudes that send every tile to the fp64 tensor path; "scaled along k": a large entry in every row of a that meets zeros
    rng = np.random.default_rng(M + N + K)
    for transa in (False, True):
        for transb in (False, True):
            a = rng.integers(-8, 9, size=(M, K)).astype(np.float64)
            b = rng.integers(-8, 9, size=(K, N)).astype(np.float64)
            c0 = rng.integers(-8, 9, size=(M, N)).astype(np.float64)
            if why == "fp64":
                a, b = a * 2.0 ** 600, b * 2.0 ** -600
            else:
                a[:, K // 2], b[K // 2] = 2.0 ** 70, 0.0
            for pitch in (padded, lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()):
                for beta in (-1.0, 0.0, 1.0):
                    c = pitch(c0)
                    g.gptq2d_internal_gemm_split(pitch(a.T if transa else a), pitch(b.T if transb else b), c, transa=transa,
                                                 transb=transb, alpha=2.0, beta=beta)
                    assert np.array_equal(c.cpu().numpy(), 2.0 * (a @ b) + beta * c0), (transa, transb, beta)


def product(g, a, b):
    c = torch.empty((a.shape[0], b.shape[1]), dtype=torch.float64, device="cuda")
    info = torch.full((4,), 9, dtype=torch.int32, device="cuda")
    g.gptq2d_internal_gemm_split(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), c, info=info)
    g.check_info(info)
    return c.cpu().numpy()


@pytest.mark.parametrize("outlier", [1e2, 1e4, 1e9])
@pytest.mark.parametrize("K", [200, 256, 1000])
@pytest.mark.parametrize("other", ["zero", "zero in some columns", "small in some columns", "there", "for half of the rows"])
def test_outlier_channels_lose_no_digits(g, K, outlier, other):
    # one k at which a is larger than elsewhere, and b is zero, small or like the rest there
    rng = np.random.default_rng(int(outlier) + K)
    M, N, k = 256, 384, K // 3
    a, b = rng.standard_normal((M, K)), rng.uniform(-0.5, 0.5, (K, N))
    a[:, k] *= outlier
    if other == "zero":
        b[k] = 0.0
    elif other == "zero in some columns":
        b[k, 100:200] = 0.0
    elif other == "small in some columns":
        b[k, 100:200] /= 50 * outlier
    elif other == "for half of the rows":
        a[:170, k] = 0.0
    want = a.astype(np.longdouble) @ b.astype(np.longdouble)
    error = np.abs(product(g, a, b) - want).astype(np.float64)
    # Entries are cut 2^-57 below the largest of their row, and rows scaled along k have their largest where the largest term of the
    # row's sums is: what that moves an entry by, 2^-57.8 (|a| + |b|) (five times in the worst of 10^5 entries), is below what a
    # chain of K fp64 additions leaves in the worst column of the row, about 2^-53 sqrt(K) (sum of (a b)^2)^(1/2).
    row = np.sqrt((a * a) @ (b * b)).max(1)[:, None]
    assert np.all(error <= 2.0 ** -53 * np.sqrt(K) * row)


@pytest.mark.parametrize("outlier", [1e3, 1e9])
def test_objective_with_an_outlier_channel_of_integers(g, outlier):
    m = n = 1024
    rng = np.random.default_rng(3)
    a, b = (np.triu(rng.standard_normal((k, k)) / np.sqrt(2 * k), 1) + np.eye(k) for k in (m, n))
    a[:, 300] *= outlier
    x = 4.0 * rng.standard_normal((m, n))
    x[300] = np.round(x[300])
    z = np.round(x)
    obj = g.gptq2d_objective(*(torch.from_numpy(v).cuda() for v in (x, z.astype(np.int32), a, b)))
    r = (z - x).astype(np.longdouble)
    want = float(np.square(a.astype(np.longdouble) @ r @ b.astype(np.longdouble)).sum())
    # two products of 1024 terms in fp64 (1e-16 sqrt(1024) each, twice in a square), uncorrelated over 10^6 entries; plus their sum
    assert abs(float(obj.cpu()[0]) - want) <= 1e-14 * want


def test_set_up_of_a_basis_whose_large_entries_do_not_meet(g):
    # one large entry a column, each in a row of its own: what couples two columns is 1e-8 of what their digits are spent on
    k = 1100
    rng = np.random.default_rng(4)
    a = rng.standard_normal((k, k))
    a[rng.permutation(k), np.arange(k)] += 1e8
    L, _, _, _, info = g.gptq2d_factor(torch.from_numpy(a).cuda(), None, n=1)
    g.check_info(info)
    got, want = np.tril(L.cpu().numpy(), -1), np.tril(O.feedback_factors(a, np.eye(1))[0], -1)
    # Gram, factor and inverse in fp64 with contractions of 1100, against the same in the oracle
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("ea,eb", [(-510, -505), (-1000, 900), (-1045, 1000), (600, -600), (700, 200), (500, 510)])
def test_extreme_magnitudes(g, ea, eb):
    # rows whose scales multiply to a subnormal number or to infinity, rows of subnormal numbers
    rng = np.random.default_rng(ea + 2000)
    a, b = rng.standard_normal((140, 100)), rng.uniform(-0.5, 0.5, (100, 150))
    a[3], b[:, 9] = 0.0, 0.0
    a, b = np.ldexp(a, ea), np.ldexp(b, eb)
    want = a.astype(np.longdouble) @ b.astype(np.longdouble)
    # 1e-16 sqrt(100) of the largest entry, and subnormal sums: half of 2^-1074 a term
    bound = 4e-15 * np.abs(want).max() + 100 * 2.0 ** -1074
    assert np.abs(want).max() < 2.0 ** 1023 and np.all(np.abs(product(g, a, b) - want) <= bound)


def test_constant_entries_with_all_digits_at_an_end_of_their_range(g):
    # K at its limit; every residue is the same along k, so that its sums are K times a square
    K = 16384
    low = sum(256.0 ** -d for d in range(2, 8))
    for x, y in ((126 / 256 + 127 * low, 126 / 256 + 127 * low), (-126 / 256 - 128 * low, 126 / 256 + 127 * low),
                 (-126 / 256 - 128 * low, -126 / 256 - 128 * low)):
        got = product(g, np.full((130, K), x), np.full((K, 5), y))
        assert np.max(np.abs(got - K * x * y)) <= 2.0 ** -50 * abs(K * x * y)


@pytest.mark.parametrize("columns", [128, 256])
@pytest.mark.parametrize("K", [1024, 1025, 16384])
def test_the_largest_sums_of_residues(g, K, columns):
    # For every modulus p, entries that are (p - 1) / 2 or its negative modulo p: sums of K ((p - 1) / 2)^2 of either sign, the largest that are reduced
    # (by one formula up to K = 1024 and another one above).  A residue that is wrong puts S off by a multiple of P / p, 2^117 and more.
    p = [256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193]
    rng = np.random.default_rng(K)

    def operand():
        # integers from 2^54 to 2^55 that are multiples of four (53 bits), a row for either sign of every modulus; all of one binary order, so that
        # scaling along k and rows' scales leave them as they are
        rows = []
        for q in p:
            for r in ((q - 1) // 2, -((q - 1) // 2)) if q % 2 else (124, -128):
                if q % 2:
                    y = rng.integers(2 ** 52, int(1.94 * 2 ** 52), size=K)
                    x = 4 * (y + (r * pow(4, -1, q) - y) % q)
                else:
                    x = rng.integers(2 ** 46, int(1.94 * 2 ** 46), size=K) * 256 + r
                assert np.all((x - r) % q == 0) and np.all(x % 4 == 0)
                rows.append(x.astype(np.float64))
        return np.array(rows)
    a, b = operand(), operand().T.copy()
    want = a.astype(np.longdouble) @ b.astype(np.longdouble)
    g.gptq2d_internal_test_hook(9, columns)
    try:
        got = product(g, a, b)
    finally:
        g.gptq2d_internal_test_hook(9, 0)
    # K terms of 2^108 and more, each sum rounded once
    assert np.max(np.abs(got / want - 1)) <= 2.0 ** -52


@pytest.mark.parametrize("k", [1100, 2200])
def test_set_up_keeps_its_digits_under_channel_scales(g, k):
    # Channel j scaled by 2^e_j scales L[i, j] by 2^(e_j - e_i), exactly.  Scales over 60 binary orders: without the scaling of the
    # products of the inverse along k their digits would be spent on them.
    rng = np.random.default_rng(k)
    s = rng.standard_normal((2 * k, k))
    a = np.linalg.cholesky(s.T @ s / (2 * k)).T
    e = rng.integers(-30, 31, size=k)
    plain, scaled = (g.gptq2d_factor(torch.from_numpy(np.ascontiguousarray(v)).cuda(), None, n=1) for v in (a, np.ldexp(a, e)))
    g.check_info(plain[4])
    g.check_info(scaled[4])
    L = plain[0].cpu().numpy()
    # against the oracle's: two fp64 factorisations of a Gram of condition 34 (1e-15 each measured)
    assert np.max(np.abs(L - O.feedback_factors(a, np.eye(1))[0])) <= 1e-13
    back = np.ldexp(scaled[0].cpu().numpy(), e[:, None] - e[None, :])
    assert np.max(np.abs(back - L)) <= 1e-14
    d = scaled[2].cpu().numpy() / np.ldexp(plain[2].cpu().numpy(), 2 * e)
    assert np.max(np.abs(d - 1.0)) <= 1e-14


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


def test_infinities_and_nans_go_where_fp64_takes_them(g):
    rng = np.random.default_rng(2)
    a, b = rng.standard_normal((300, 400)), rng.standard_normal((400, 260))
    a[7, 3], a[200, 399], a[130, 64] = np.inf, np.nan, -np.inf
    b[3, :100], b[64, 5], b[399, 128:] = 0.0, np.inf, 0.0
    a[:, 320:384] = 0.0                                        # a chunk without an entry in a, but with one in b
    b[330, 140] = np.inf
    with np.errstate(invalid="ignore"):
        want = a @ b
    got = product(g, a, b)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    inf = np.isinf(want)
    assert np.array_equal(got[inf], want[inf]) and np.isnan(got).any() and inf.any()
    fine = np.isfinite(want)
    assert np.max(np.abs(got[fine] - want[fine])) < 1e-12


@pytest.mark.parametrize("columns", [128, 256])
@pytest.mark.parametrize("M,N,K", [(256, 256, 128), (255, 257, 1024), (257, 129, 1025), (513, 385, 1152), (130, 650, 2304)])
def test_tiles_of_both_widths(g, columns, M, N, K):
    # edges of tiles, of the halves of a pair and of stages of 128 and 256 k; both sides of K = 1024, where the reduction of the sums
    # changes.  Integers of 20 bits: sums below 2^52 and multiples of 2^60 of the scaled product, so exact.  Triangles: tiles in reverse order.
    rng = np.random.default_rng(M + N + K)
    a = rng.integers(-2 ** 20, 2 ** 20, size=(M, K)).astype(np.float64)
    b = rng.integers(-2 ** 20, 2 ** 20, size=(K, N)).astype(np.float64)
    g.gptq2d_internal_test_hook(9, columns)
    try:
        for x, y in ((a, b), (np.triu(a), b), (np.tril(a), np.tril(b)), (a, np.triu(b))):
            assert np.array_equal(product(g, x, y), x @ y)
    finally:
        g.gptq2d_internal_test_hook(9, 0)


@pytest.mark.parametrize("M,K", [(32, 64), (33, 65), (70, 300)])
def test_digits_at_the_ends_of_their_range(g, M, K):
    # entries whose seven balanced base-256 digits are mostly -128, 127, 0 and +-1, where a residue is largest before it is reduced; the lowest
    # digit 0 or -128, so 49 bits.  Against columns with a single one: sums of one term, multiples of 2^61 of the scaled product, so exact.
    rng = np.random.default_rng(M + K)
    digits = rng.choice([-128, -127, 127, 126, -1, 0, 1], size=(7, M, K))
    digits[0] = rng.choice([0, -128], size=(M, K))
    digits[6] = rng.choice([-126, 126, 0], size=(M, K))
    digits[6, :, 0] = 126                                    # every row's scale is that of 56 bits
    a = sum(digits[j].astype(np.int64) << (8 * j) for j in range(7)).astype(np.float64)
    where = rng.integers(0, K, size=150)
    b = np.zeros((K, 150))
    b[where, np.arange(150)] = 1.0
    assert np.array_equal(product(g, a, b), a[:, where])
    assert np.array_equal(product(g, b.T.copy(), a.T.copy()), a[:, where].T)


@pytest.mark.parametrize("columns", [128, 256])
def test_a_sum_is_rounded_once(g, columns):
    # multiples of 2^-53 below 1/2 lose nothing as integers, so what is left is putting the sums together: one rounding, not two (1.41)
    rng = np.random.default_rng(columns)
    M, N, K = 300, 260, 700
    a, b = rng.uniform(-0.5, 0.5, (M, K)), rng.uniform(-0.5, 0.5, (K, N))
    want = a.astype(np.longdouble) @ b.astype(np.longdouble)
    g.gptq2d_internal_test_hook(9, columns)
    try:
        got = product(g, a, b)
    finally:
        g.gptq2d_internal_test_hook(9, 0)
    once = np.linalg.norm((want.astype(np.float64) - want).astype(np.float64))
    # (the weights' 80 bits and 2^-64 sqrt(K) of the reference are a hundredth of it)
    assert np.linalg.norm((got - want).astype(np.float64)) <= 1.05 * once
