"""The set-up at the orders where its small kernels change over (64, 96, 128 rows a block) and where the levels of the triangular
inverse have an odd last block, against the oracle's factors."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2607_27042_b200 import workloads as W

pytestmark = pytest.mark.gpu


def check(got, want):
    # two fp64 factorisations of Grams of condition below 1e4: 1e-9 of the largest entry, as everywhere in these tests
    assert np.max(np.abs(got - want)) <= 1e-9 * np.max(np.abs(want))


@pytest.mark.parametrize("batched", [True, False])
def test_orders_around_the_class_boundaries(batched):
    from paper_2607_27042_b200 import gptq2d as g
    shapes = [(1, 16), (17, 48), (63, 64), (65, 95), (96, 97), (127, 128), (33, 80), (112, 90)]
    cases = [W.general_bases(m, n, 40 + i) for i, (m, n) in enumerate(shapes)]
    if batched:
        As, Bs = [torch.from_numpy(c[1]).cuda() for c in cases], [torch.from_numpy(c[2]).cuda() for c in cases]
        Ls, Us, dLs, dUs, info = g.gptq2d_factor_batched(As, Bs)
        g.check_info(info)
        got = list(zip(Ls, Us))
    else:
        got = []
        for c in cases:
            L, U, _, _, info = g.gptq2d_factor(torch.from_numpy(c[1]).cuda(), torch.from_numpy(c[2]).cuda())
            g.check_info(info)
            got.append((L, U))
    for c, (L, U) in zip(cases, got):
        wantL, wantU, _, _ = O.feedback_factors(c[1], c[2])
        check(L.cpu().numpy(), wantL)
        check(U.cpu().numpy(), wantU)


@pytest.mark.parametrize("k", [128 * 3 + 4, 128 * 5, 128 * 7 + 100, 128 * 9 + 1, 2200])
def test_odd_last_blocks_of_the_inverse(k):
    from paper_2607_27042_b200 import gptq2d as g
    _, A, _ = W.gaussian_like(k, 8, seed=k, samples=2 * k)
    L, _, _, _, info = g.gptq2d_factor(torch.from_numpy(A).cuda(), None, n=1)
    g.check_info(info)
    check(L.cpu().numpy(), O.feedback_factors(A, np.eye(1))[0])
