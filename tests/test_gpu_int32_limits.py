"""Z next to the ends of int32: what fits is returned, what does not is reported and saturated."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TOP = 2.0 ** 31
FITS = [(TOP - 2.6, 2 ** 31 - 3), (TOP - 1.5, 2 ** 31 - 2), (TOP - 0.75, 2 ** 31 - 1), (np.nextafter(TOP - 0.5, 0.0), 2 ** 31 - 1),
        (-TOP + 0.75, -2 ** 31 + 1), (-TOP + 0.5, -2 ** 31), (np.nextafter(-TOP, 0.0), -2 ** 31)]
LIES_BEYOND = [(TOP - 0.5, 2 ** 31 - 1), (TOP - 0.4, 2 ** 31 - 1), (np.nextafter(TOP, 0.0), 2 ** 31 - 1), (TOP, 2 ** 31 - 1),
               (TOP + 0.3, 2 ** 31 - 1), (1e300, 2 ** 31 - 1), (-TOP, -2 ** 31), (-TOP - 0.6, -2 ** 31), (-1e300, -2 ** 31)]


def sweep(batched, m, n, i, j, value):
    from paper_2607_27042_b200 import gptq2d as g
    X = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    X[i, j] = value
    L, U = (torch.eye(k, dtype=torch.float64, device="cuda") for k in (m, n))
    if batched:
        Zs, _, _, info = g.gptq2d_round_batched([X], [L], [U])
        Z = Zs[0]
    else:
        Z, _, _, info = g.gptq2d_round(X, L, U)
    return Z.cpu().numpy(), info.cpu().tolist()


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("m,n,i,j", [(1, 1, 0, 0), (8, 8, 7, 7), (70, 130, 4, 0), (70, 130, 69, 129), (130, 70, 66, 68)])
def test_values_at_the_ends_of_int32(batched, m, n, i, j):
    for values, reported in ((FITS, False), (LIES_BEYOND, True)):
        for value, want in values:
            Z, info = sweep(batched, m, n, i, j, value)
            assert Z[i, j] == want, (value, Z[i, j], info)
            assert info == ([7, i, j, 0] if reported else [0, 0, 0, 0]), (value, info)
            Z[i, j] = 0
            assert not Z.any(), value
