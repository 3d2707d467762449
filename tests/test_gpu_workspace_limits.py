"""Workspaces without room for what only makes a call faster (the residue planes of large products, the bookkeeping of a sweep in
blocks): accepted, with the same results; a byte less is refused."""
import numpy as np
import pytest
import torch

from paper_2607_27042_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture()
def g():
    from paper_2607_27042_b200 import gptq2d
    yield gptq2d
    gptq2d.gptq2d_internal_test_hook(7, 0)


def up(x, a=256):
    return -(-x // a) * a


def side(k):
    """Gram, inverse, product buffer and pivots of one side."""
    return up(3 * 8 * up(k, 16) ** 2 + 8 * up(k, 32) + 256)


def ws(nbytes):
    return torch.full((nbytes,), 0xff, dtype=torch.uint8, device="cuda")


def refused(g, call, nbytes):
    with pytest.raises(g.Gptq2dError) as e:
        call(ws(nbytes))
    assert e.value.status == 2


def test_set_up(g):
    m, n = 1300, 1031
    _, A, B = W.gaussian_like(m, n, 5, samples=2 * m)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    least = side(m) + side(n)
    assert g.gptq2d_factor_workspace_bytes(m, n) > least
    want = g.gptq2d_factor(dA, dB)
    got = g.gptq2d_factor(dA, dB, workspace=ws(least))
    own = sum(2 * up(8 * k * k) + up(8 * k) for k in (m, n))
    rev_want = g.gptq2d_factor_reverse(dA, dB)
    rev = g.gptq2d_factor_reverse(dA, dB, workspace=ws(own + least))
    for a, b in ((got, want), (rev, rev_want)):
        g.check_info(a[4])
        # two fp64 factorisations of well-conditioned Grams: 1e-12 is a thousand roundings
        for x, y in zip(a[:4], b[:4]):
            assert float((x - y).abs().max()) <= 1e-12 * float(y.abs().max())
    refused(g, lambda w: g.gptq2d_factor(dA, dB, workspace=w), least - 256)
    refused(g, lambda w: g.gptq2d_factor_reverse(dA, dB, workspace=w), own + least - 256)


def test_set_up_with_room_for_some_planes(g):
    # each side's updates of rank 768 need a tenth of the room for all products, its largest joins all of it
    m, n = 4700, 4610
    A, B = (torch.randn(k, k, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(k)) / (4 * k) ** 0.5 +
            torch.eye(k, dtype=torch.float64, device="cuda") for k in (m, n))
    least, most = side(m) + side(n), g.gptq2d_factor_workspace_bytes(m, n)
    out = []
    for share in (0.0, 0.2, 0.45, 1.0):
        got = g.gptq2d_factor(A, B, workspace=ws(least + int(share * (most - least))))
        g.check_info(got[4])
        out.append(got)
    for got in out[1:]:
        for x, y in zip(got[:4], out[0][:4]):
            # two fp64 factorisations of Grams of condition below 100
            assert float((x - y).abs().max()) <= 1e-12 * float(y.abs().max())
    # every share takes products that the one before had no room for
    for x, y in zip(out, out[1:]):
        assert not torch.equal(x[0], y[0]) and not torch.equal(x[1], y[1])


def test_set_up_batched(g):
    shapes = [(1100, 40), (1030, 1024), (60, 70)]
    cases = [W.gaussian_like(m, n, 6 + i, samples=2 * max(m, n)) for i, (m, n) in enumerate(shapes)]
    As, Bs = ([torch.from_numpy(c[i]).cuda() for c in cases] for i in (1, 2))
    want = g.gptq2d_factor_batched(As, Bs)
    outs = [[torch.empty_like(t) for t in want[i]] for i in range(4)]
    problems = g.make_factor_problems(As, Bs, *outs)
    # a table, and two problems of the blocked route side by side, each in a slot of the larger one's size
    table = g.gptq2d_factor_batched_workspace_bytes(problems) - 2 * max(g.gptq2d_factor_workspace_bytes(m, n) for m, n in shapes[:2])
    slots = 2 * max(side(m) + side(n) for m, n in shapes[:2])
    info = torch.zeros(4, dtype=torch.int32, device="cuda")
    g.gptq2d_factor_batched(problems=problems, workspace=ws(table + slots), info=info)
    g.check_info(info)
    for xs, ys in zip(outs, want[:4]):
        for x, y in zip(xs, ys):
            assert float((x - y).abs().max()) <= 1e-12 * float(y.abs().max())
    refused(g, lambda w: g.gptq2d_factor_batched(problems=problems, workspace=w, info=info), table + slots - 256)


def test_objective(g):
    m, n = 1024, 1030
    X, A, B = W.gaussian_like(m, n, 7)
    args = [torch.from_numpy(v).cuda() for v in (X, np.round(X).astype(np.int32), A, B)]
    least = up(2 * 8 * m * up(n, 16) + up(8 * (-(-m // 128)) * (-(-n // 128))) + 256)
    assert g.gptq2d_objective_workspace_bytes(m, n) > least
    want, got = float(g.gptq2d_objective(*args)[0]), float(g.gptq2d_objective(*args, workspace=ws(least))[0])
    assert abs(got - want) <= 1e-13 * want
    refused(g, lambda w: g.gptq2d_objective(*args, workspace=w), least - 256)


@pytest.mark.parametrize("entry", ["round", "reverse", "f32in", "host"])
def test_sweep(g, entry):
    m, n = 400, 300
    rng = np.random.default_rng(8)
    X = 4.0 * rng.standard_normal((m, n))
    L, U = np.tril(rng.standard_normal((m, m)), -1) / m, np.triu(rng.standard_normal((n, n)), 1) / n
    if entry == "reverse":
        L, U = L.T.copy(), U.T.copy()
    X, L, U = (torch.from_numpy(v) for v in (X, L, U))
    if entry == "f32in":
        X, L, U = X.float(), L.float(), U.float()
    X, L, U = (v.pin_memory() if entry == "host" else v.cuda() for v in (X, L, U))
    call, size = {"round": (g.gptq2d_round, g.gptq2d_round_workspace_bytes),
                  "reverse": (g.gptq2d_round_reverse, g.gptq2d_round_reverse_workspace_bytes),
                  "f32in": (g.gptq2d_round_f32in, g.gptq2d_round_f32in_workspace_bytes),
                  "host": (g.gptq2d_round_host, g.gptq2d_round_host_workspace_bytes)}[entry]
    least = size(m, n)
    want = call(X, L, U)[0].cpu()
    g.gptq2d_internal_test_hook(7, 129)                # from now on these matrices are swept in blocks, if there is room
    assert size(m, n) > least
    assert torch.equal(call(X, L, U)[0].cpu(), want)
    assert torch.equal(call(X, L, U, workspace=ws(least))[0].cpu(), want)
    refused(g, lambda w: call(X, L, U, workspace=w), least - 256)
