"""The small parity cases once more under the CHECKED build of the library (libgptq2d_checked.so,
-DGPTQ2D_CHECKED): the computed indexes of every shared- and global-memory access of the tiled sweep, and the main ones
of its DMMA tile loop, of the blocked sweep and of the tiles of the int8 products, are range-checked on the device, and a violation comes back through
the status words as GPTQ2D_ERR_CHECK (nothing traps).  compute-sanitizer is not available where this library
is developed; this is its stand-in.  Runs in a process of its own so that the two builds never share one."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import sys
sys.path.insert(0, %r)
sys.path.insert(0, %r)
import numpy as np, torch
import oracle as O
from oracle import cref
from certify import certified_case
from paper_2607_27042_b200 import gptq2d as g, workloads as W
assert g.library_path().endswith("libgptq2d_checked.so")
# the check itself: a deliberately bad index must be recorded (status 10, site, index, limit) and redirected to 0
probe = torch.full((5,), -1, dtype=torch.int32, device="cuda")
g.gptq2d_internal_test_hook(5, probe.data_ptr())
torch.cuda.synchronize()
assert probe.cpu().tolist() == [10, 999, 7, 3, 0], probe.cpu().tolist()

def draw(m, n):
    def d(seed):
        X, A, B = W.general_bases(m, n, seed)
        L, U, _, _ = O.feedback_factors(A, B)
        return X, L, U
    return d

cases = []
for k, (m, n) in enumerate([(1, 1), (17, 5), (65, 63), (129, 257), (200, 75), (257, 130), (300, 515), (3, 700)]):
    (X, L, U), ref, _ = certified_case(draw(m, n), cref.nested, 50 + k)
    dX, dL, dU = (torch.from_numpy(a).cuda() for a in (X, L, U))
    Z, E, mm, info = g.gptq2d_round(dX, dL, dU, want_E=True, want_margin=True)
    torch.cuda.synchronize()
    g.check_info(info)                                   # raises on GPTQ2D_ERR_CHECK (status 10)
    assert np.array_equal(Z.cpu().numpy().astype(np.int64), ref["Z"]), (m, n)
    g.gptq2d_internal_test_hook(7, 129)                  # the same in 2 x 2 blocks, where there are two tiles each way
    Z, E, mm, info = g.gptq2d_round(dX, dL, dU, want_E=True, want_margin=True)
    torch.cuda.synchronize()
    g.gptq2d_internal_test_hook(7, 0)
    g.check_info(info)
    assert np.array_equal(Z.cpu().numpy().astype(np.int64), ref["Z"]), (m, n)
    for w in (17, 64):
        Zb, _, _, ib = g.gptq2d_round_blocked(dX, dL, dU, w)
        torch.cuda.synchronize()
        g.check_info(ib)
        assert np.array_equal(Zb.cpu().numpy().astype(np.int64), ref["Z"]), (m, n, w)
    cases.append((dX, dL, dU, ref["Z"]))
Zs, _, _, info = g.gptq2d_round_batched([c[0] for c in cases], [c[1] for c in cases], [c[2] for c in cases])
torch.cuda.synchronize()
g.check_info(info)
for z, c in zip(Zs, cases):
    assert np.array_equal(z.cpu().numpy().astype(np.int64), c[3])
hX, hL, hU = (c.cpu().pin_memory() for c in cases[6][:3])
hZ, hinfo = g.gptq2d_round_host(hX, hL, hU)
assert np.array_equal(hZ.numpy().astype(np.int64), cases[6][3])
# a product on the int8 tensor cores, ragged, odd pitches; the second time its tiles are computed in fp64 (extreme magnitudes)
a = torch.randint(-8, 9, (257, 191), device="cuda").double()
b = torch.randint(-8, 9, (191, 131), device="cuda").double()
for scale in (1.0, 2.0 ** 600):
    a, b = a * scale, b / scale
    c = torch.ones((257, 131), dtype=torch.float64, device="cuda")
    info = torch.zeros(4, dtype=torch.int32, device="cuda")
    g.gptq2d_internal_gemm_split(a, b, c, beta=1.0, info=info)
    g.check_info(info)
    assert np.array_equal(c.cpu().numpy(), a.cpu().numpy() @ b.cpu().numpy() + 1.0)
print("checked build: %%d cases clean" %% len(cases))
"""

CELLS = r"""
import sys
sys.path.insert(0, %r)
sys.path.insert(0, %r)
import numpy as np, torch
from paper_2607_27042_b200 import gptq2d as g
assert g.library_path().endswith("libgptq2d_checked.so")
rng = np.random.default_rng(3)

def padded(a, extra):
    buf = torch.full((a.shape[0], a.shape[1] + extra), float("nan"), dtype=torch.float64, device="cuda")
    buf[:, :a.shape[1]] = torch.from_numpy(a).cuda()
    return buf[:, :a.shape[1]]

# far parts in both directions, cells at both edges, a value that does not fit; operands in pieces of 16 and of 8 bytes
for m, n in [(545, 399), (399, 545), (512, 640)]:
    X = 4.0 * rng.standard_normal((m, n))
    L, U = np.tril(rng.standard_normal((m, m)), -1) / m, np.triu(rng.standard_normal((n, n)), 1) / n
    out = []
    for extra in (0, 1):
        E = padded(np.zeros((m, n)), 3)
        for order, less in ((1 << 30, 0), (129, 0), (129, 1)):
            g.gptq2d_internal_test_hook(7, order)
            size = g.gptq2d_round_workspace_bytes(m, n)
            if less:                                     # no room for the planes between blocks: in free rows, in pieces
                m0, n0 = ((-(-k // 128) + 1) // 2 * 128 for k in (m, n))
                size -= 16 * (m0 + n0) * max(m0, n0)
                assert (g.gptq2d_internal_round_products(m, n, size) > 4) == (m < n)      # (the rows below a tall block are too few)
            ws = torch.full((size,), 0xff, dtype=torch.uint8, device="cuda")
            Z, _, _, info = g.gptq2d_round(padded(X, extra), padded(L, m %% 2 + extra), padded(U, n %% 2 + extra), E=E, workspace=ws)
            g.check_info(info)
            out.append(Z.cpu())
    assert all(torch.equal(z, out[0]) for z in out)
    X[m - 1, n - 1] = 1e300
    info = g.gptq2d_round(padded(X, 0), padded(L, 0), padded(U, 0))[3].cpu().tolist()
    assert info[0] not in (0, 10), info
g.gptq2d_internal_test_hook(7, 0)
print("checked build: cells clean")
"""


def test_cells_under_the_checked_build():
    from paper_2607_27042_b200 import build
    build.build(checked=True)
    env = dict(os.environ, GPTQ2D_LIBRARY="libgptq2d_checked.so")
    r = subprocess.run([sys.executable, "-c", CELLS % (ROOT, os.path.join(ROOT, "tests"))], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "cells clean" in r.stdout


def test_small_parity_cases_under_the_checked_build():
    from paper_2607_27042_b200 import build
    build.build(checked=True)                                # no-op when the library is already there
    env = dict(os.environ, GPTQ2D_LIBRARY="libgptq2d_checked.so")
    r = subprocess.run([sys.executable, "-c", SCRIPT % (ROOT, os.path.join(ROOT, "tests"))], env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "cases clean" in r.stdout
