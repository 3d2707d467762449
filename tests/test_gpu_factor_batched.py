"""GPU parity of the batched set-up (gptq2d_factor_batched) against the CPU oracle's factors
(Section 3.1: L unit lower with (A^T A)^{-1} = L Lambda_L L^T, U unit upper with (B B^T)^{-1} = U^T Lambda_U U)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2607_27042_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_2607_27042_b200 import gptq2d
    return gptq2d


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).cuda()


def check(g, shapes, seeds, with_identity=()):
    As, Bs, refs = [], [], []
    for b, ((m, n), seed) in enumerate(zip(shapes, seeds)):
        _, A, B = W.general_bases(m, n, seed)
        if b in with_identity:
            A = None
        As.append(None if A is None else dev(A))
        Bs.append(dev(B))
        refs.append(O.feedback_factors(np.eye(m) if A is None else A, B))
    Ls, Us, dLs, dUs, info = g.gptq2d_factor_batched(As, Bs, shapes=shapes)
    torch.cuda.synchronize()
    g.check_info(info)
    for b, (L, U, lamL, lamU) in enumerate(refs):
        gl, gu = Ls[b].cpu().numpy(), Us[b].cpu().numpy()
        sc = max(1.0, np.max(np.abs(L)), np.max(np.abs(U)))
        assert np.max(np.abs(gl - L)) < 1e-9 * sc, (b, shapes[b])
        assert np.max(np.abs(gu - U)) < 1e-9 * sc, (b, shapes[b])
        assert np.allclose(dLs[b].cpu().numpy(), 1.0 / lamL, rtol=1e-9), b
        assert np.allclose(dUs[b].cpu().numpy(), 1.0 / lamU, rtol=1e-9), b
        # exact ones on the diagonal, exact zeros in the opposite triangle
        assert np.array_equal(np.tril(gl), gl) and np.array_equal(np.diag(gl), np.ones(gl.shape[0]))
        assert np.array_equal(np.triu(gu), gu) and np.array_equal(np.diag(gu), np.ones(gu.shape[0]))
    return As, Bs, Ls, Us


def test_small_sides_of_every_size_class(g):
    shapes = [(1, 1), (1, 9), (9, 1), (17, 5), (64, 64), (100, 33), (128, 128), (127, 128), (33, 100), (2, 128)]
    check(g, shapes, seeds=range(len(shapes)), with_identity=(3,))


def test_mixed_small_and_large_sides_and_agreement_with_the_single_call(g):
    shapes = [(64, 64), (200, 90), (90, 300), (129, 129), (16, 16)]
    As, Bs, Ls, Us = check(g, shapes, seeds=[10, 11, 12, 13, 14])
    for b in range(len(shapes)):
        L1, U1, _, _, info = g.gptq2d_factor(As[b], Bs[b])
        torch.cuda.synchronize()
        g.check_info(info)
        assert float((L1 - Ls[b]).abs().max()) < 1e-10 * max(1.0, float(L1.abs().max()))
        assert float((U1 - Us[b]).abs().max()) < 1e-10 * max(1.0, float(U1.abs().max()))


def test_one_large_problem_among_small_ones_and_many_large_ones(g):
    """One problem of the blocked route takes gptq2d_factor's two-stream path; several of them are spread
    over a pool of streams (more problems than streams here, so slots are reused in order)."""
    check(g, [(64, 64), (300, 200), (5, 7)], seeds=[20, 21, 22])
    shapes = [(130 + 7 * b, 129 + 5 * b) for b in range(11)] + [(33, 33)]
    check(g, shapes, seeds=range(30, 30 + len(shapes)))


def test_two_hundred_config_c0_like_pairs_feed_the_batched_sweep(g):
    """The use the entry point exists for: factors of many 64 x 64 layers in one launch, then one batched sweep;
    every Z against the oracle's plain-C nested sweep where the certificate allows it."""
    from oracle import cref
    count = 200
    Xs, As, Bs, refs = [], [], [], []
    for b in range(count):
        X, A, B = W.make_config(0, seed=b)
        Xs.append(dev(X)); As.append(dev(A)); Bs.append(dev(B))
        refs.append((X, A, B))
    Ls, Us, _, _, finfo = g.gptq2d_factor_batched(As, Bs)
    Zs, _, mm, info = g.gptq2d_round_batched(Xs, Ls, Us, want_margin=True)
    torch.cuda.synchronize()
    g.check_info(finfo)
    g.check_info(info)
    checked = 0
    for b in range(0, count, 8):
        X, A, B = refs[b]
        L, U, _, _ = O.feedback_factors(A, B)
        ref = cref.nested(X, L, U)
        margin, _ = O.certificate_margin(X, ref["Z"], L, U)
        if margin >= 1e-9:
            assert np.array_equal(Zs[b].cpu().numpy().astype(np.int64), ref["Z"]), b
            assert abs(float(mm.cpu()[b]) - margin) < 1e-9
            checked += 1
    assert checked >= 15


def test_a_singular_basis_names_its_problem_and_the_others_are_still_factorised(g):
    shapes = [(20, 20), (30, 12), (40, 40)]
    As, Bs = [], []
    for b, (m, n) in enumerate(shapes):
        _, A, B = W.general_bases(m, n, 50 + b)
        if b == 1:
            A[:, 7] = 0.0                      # singular A: its Gram has a zero pivot
        As.append(dev(A)); Bs.append(dev(B))
    Ls, Us, _, _, info = g.gptq2d_factor_batched(As, Bs)
    torch.cuda.synchronize()
    vals = info.cpu().tolist()
    assert vals[0] == 5 and vals[2] == 0 and vals[3] == 1          # NOT_SPD, side A, problem 1
    for b in (0, 2):
        _, A, B = W.general_bases(*shapes[b], 50 + b)
        L, U, _, _ = O.feedback_factors(A, B)
        assert np.max(np.abs(Ls[b].cpu().numpy() - L)) < 1e-9 * max(1.0, np.max(np.abs(L)))
        assert np.max(np.abs(Us[b].cpu().numpy() - U)) < 1e-9 * max(1.0, np.max(np.abs(U)))


def test_the_multi_stream_set_up_is_bit_identical_to_the_one_stream_set_up(g):
    """With both bases given, gptq2d_factor runs the two sides on two streams and each side's chain of
    diagonal blocks ahead of its large updates on a third and fourth; with one basis it runs on the
    caller's stream alone.  Same kernels, same operands, so the outputs must agree bit for bit, run after
    run (a missing dependency between the streams would show up here)."""
    torch.manual_seed(3)
    for k, kb, reps in [(300, 337, 20), (640, 513, 10), (1500, 1200, 4)]:
        A = torch.randn(k, k, dtype=torch.float64, device="cuda") / k ** 0.5 + torch.eye(k, dtype=torch.float64, device="cuda")
        B = torch.randn(kb, kb, dtype=torch.float64, device="cuda") / kb ** 0.5 + torch.eye(kb, dtype=torch.float64, device="cuda")
        L0, _, dL0, _, i0 = g.gptq2d_factor(A, None, n=1)
        _, U0, _, dU0, i1 = g.gptq2d_factor(None, B, m=1)
        torch.cuda.synchronize()
        g.check_info(i0)
        g.check_info(i1)
        for _ in range(reps):
            L, U, dL, dU, info = g.gptq2d_factor(A, B)
            torch.cuda.synchronize()
            g.check_info(info)
            assert torch.equal(L, L0) and torch.equal(U, U0) and torch.equal(dL, dL0) and torch.equal(dU, dU0), k


@pytest.mark.parametrize("e", [470, -490])
@pytest.mark.parametrize("k", [1, 16, 17, 64, 97, 128, 150])
def test_diagonal_blocks_near_the_ends_of_the_range(g, k, e):
    # pivots of 2^940 and 2^-980, where the approximate inverses are not taken; a power of two changes no digit of L but for those
    rng = np.random.default_rng(k)
    a = rng.standard_normal((k, k)) / np.sqrt(4 * k) + np.eye(k)
    plain, scaled = (g.gptq2d_factor(dev(v), None, n=1) for v in (a, np.ldexp(a, e)))
    g.check_info(plain[4])
    g.check_info(scaled[4])
    # two factorisations of a Gram of condition below 100: 128 roundings of 1e-16 times that
    assert float((scaled[0] - plain[0]).abs().max()) <= 2e-12
    assert np.max(np.abs(np.ldexp(scaled[2].cpu().numpy(), -2 * e) / plain[2].cpu().numpy() - 1.0)) <= 2e-12


@pytest.mark.parametrize("k,i,j", [(40, 5, 6), (40, 0, 15), (40, 18, 29), (40, 33, 39), (128, 112, 127), (96, 7, 13)])
def test_a_repeated_channel_is_a_zero_pivot(g, k, i, j):
    # two equal columns of one block of sixteen: what is left of the first after the second is zero, not a rounding error of either sign
    for seed in range(4):
        a = np.random.default_rng(seed).standard_normal((k, k))
        a[:, i] = a[:, j]
        assert g.gptq2d_factor_batched([dev(a)], [dev(np.eye(1))])[4].cpu().tolist() == [5, i, 0, 0]


@pytest.mark.parametrize("scaled", [False, True])
@pytest.mark.parametrize("m,n", [(4352, 4353), (4480, 4481), (5000, 3750), (4097, 5120), (40, 5889), (5760, 100)])
def test_loops_with_one_and_two_levels_agree(g, m, n, scaled):
    # both sides of the rule that chooses the loop by the orders of a call's two sides, last outer blocks of one to six block rows; against
    # the calls with one basis, which take the loop with one level
    torch.manual_seed(m)
    A, B = (torch.randn(k, k, dtype=torch.float64, device="cuda") / (4 * k) ** 0.5 + torch.eye(k, dtype=torch.float64, device="cuda") for k in (m, n))
    # channels of log-normal scales: column j of A, row j of B; entry (i, j) of L then is s_j / s_i times as large, (i, j) of U s_i / s_j
    a, b = (torch.exp(torch.randn(k, dtype=torch.float64, device="cuda")) if scaled else torch.ones(k, dtype=torch.float64, device="cuda") for k in (m, n))
    A, B = A * a, B * b[:, None]
    L, U, dL, dU, info = g.gptq2d_factor(A, B)
    L1, _, dL1, _, i0 = g.gptq2d_factor(A, None, n=1)
    _, U1, _, dU1, i1 = g.gptq2d_factor(None, B, m=1)
    for i in (info, i0, i1):
        g.check_info(i)
    # the same sums in pieces of 128 and 768 k: ten times what is measured, 1.1e-16 for entries of 0.1 and less and 1.8e-15 for squared pivots
    assert float(((L - L1) * a[:, None] / a).abs().max()) <= 1e-15 and float(((U - U1) * b / b[:, None]).abs().max()) <= 1e-15
    assert float((dL / dL1 - 1).abs().max()) <= 1.8e-14 and float((dU / dU1 - 1).abs().max()) <= 1.8e-14


@pytest.mark.parametrize("k", [897, 1024, 1025, 1500, 3000, 4100])
def test_the_inverse_in_two_parts_is_bit_identical_to_the_one_in_one(g, k):
    # eight block rows and more: the lower rows' inverse is put together beneath the factorisation of the upper ones; last levels of two blocks
    # and of three, last blocks of one row, four and a whole one.  The same products as in the calls with one basis.
    torch.manual_seed(k)
    A, B = (torch.randn(j, j, dtype=torch.float64, device="cuda") / (4 * j) ** 0.5 + torch.eye(j, dtype=torch.float64, device="cuda") for j in (k, 200))
    L1, _, dL1, _, i1 = g.gptq2d_factor(A, None, n=1)
    _, U2, _, dU2, i2 = g.gptq2d_factor(None, A, m=1)
    for _ in range(3):
        L, _, dL, _, ia = g.gptq2d_factor(A, B)
        _, U, _, dU, ib = g.gptq2d_factor(B, A)
        for i in (i1, i2, ia, ib):
            g.check_info(i)
        assert torch.equal(L, L1) and torch.equal(dL, dL1) and torch.equal(U, U2) and torch.equal(dU, dU2)


@pytest.mark.parametrize("k", [1100, 1990, 2300, 4090])
def test_the_planes_serve_one_stream_at_a_time(g, k):
    # with every product on the int8 tensor cores both streams of the inverse's parts use the planes all the time: bit for bit the call with one
    # basis, which has one stream
    torch.manual_seed(k)
    A, B = (torch.randn(j, j, dtype=torch.float64, device="cuda") / (4 * j) ** 0.5 + torch.eye(j, dtype=torch.float64, device="cuda") for j in (k, 1030))
    plain = g.gptq2d_factor(A, None, n=1)
    g.gptq2d_internal_test_hook(10, 1)
    try:
        L1, _, dL1, _, i1 = g.gptq2d_factor(A, None, n=1)
        _, U2, _, dU2, i2 = g.gptq2d_factor(None, A, m=1)
        for _ in range(5):
            L, _, dL, _, ia = g.gptq2d_factor(A, B)
            _, U, _, dU, ib = g.gptq2d_factor(B, A)
            for i in (i1, i2, ia, ib):
                g.check_info(i)
            assert torch.equal(L, L1) and torch.equal(dL, dL1) and torch.equal(U, U2) and torch.equal(dU, dU2)
    finally:
        g.gptq2d_internal_test_hook(10, 0)
    # and with most of them on the fp64 tensor path: a Gram of condition below 100, k roundings of 2^-53 times that
    assert not torch.equal(plain[0], L1) and float((plain[0] - L1).abs().max()) <= k * 2.0 ** -53 * 100


def test_reciprocals_and_quotients_of_the_pivots(g):
    # d over the whole range in which the approximate inverse is taken, significands next to powers of two among them; x up to 2 d
    rng = np.random.default_rng(0)
    n = 200000
    ends = np.arange(1, 65) * 2.0 ** -52
    significands = np.concatenate([rng.uniform(1.0, 2.0, n), np.repeat([1.0], 64), 1.0 + ends, 2.0 - ends])
    e = rng.integers(-960, 900, size=significands.size)
    d = np.ldexp(significands, e)
    x = np.ldexp(rng.uniform(-2.0, 2.0, d.size), np.maximum(e + rng.integers(-40, 1, size=d.size), -960))
    x[::7] = d[::7]
    rcp, quotient = (t.cpu().numpy() for t in g.gptq2d_internal_chol_division(dev(x), dev(d)))
    w = np.longdouble
    dw, u = d.astype(w), 2.0 ** -53

    def off(got, want):
        return float(np.max(np.abs(got.astype(w) / want - 1)))
    # the last step's correction is right to 2^-76: half a unit in the last place, and as much of the division
    assert off(rcp, 1 / dw) <= 1.001 * u
    some = x != 0.0
    assert off(quotient[some], (x.astype(w) / dw)[some]) <= 1.001 * u and np.all(quotient[::7] == 1.0)
    # next to a division: a neighbour at most
    assert np.max(np.abs(rcp * d - 1.0)) <= 2 * u and np.all(np.abs(quotient - x / d) <= 2 * u * np.abs(x / d))
