"""The FP64 estimate of one pair against the exact rational value of its own neighbour counts:
psi(n) = H(n-1) - gamma, so the estimate is a sum of harmonic numbers in which gamma cancels.
Bound, with u the unit in the last place of psi(M): every digamma value is within u of the exact
one, and a mean of them no further off; the estimate holds four of them (k, M and the two means).
Its operations on values up to 2 psi(M), the sum's conversion, the division by M, one addition and one
subtraction, add at most u each, 1/k and its subtraction less than u together: 9 u."""
import math
from decimal import Decimal, getcontext

import numpy as np
import pytest

from test_gpu_exact import load

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alg", [1, 2])
@pytest.mark.parametrize("M", [7, 8, 9, 16, 17, 31, 32, 33, 64, 65, 100, 333, 1000, 2049, 4096])
def test_estimate_of_a_pair_is_fp64(ndf_mod, ctx, M, alg):
    getcontext().prec = 40
    H = [Decimal(0)]
    for i in range(1, M + 1):
        H.append(H[-1] + Decimal(1) / i)
    rng = np.random.default_rng(M)
    s = rng.normal(size=(M, 1, 1, 1))
    w = np.linspace(0.0, 0.999, 12)
    f = (w * s + np.sqrt(1 - w * w) * rng.normal(size=(M, 1, 1, 12))).astype(np.float32)
    fid = load(ndf_mod, ctx, f)
    psi_M = float(H[M - 1]) - 0.5772156649015329
    bound = 9 * 2.0 ** (math.floor(math.log2(psi_M)) - 52)
    a, b = np.empty(M, np.float32), np.empty(M, np.float32)
    nx, ny = np.empty(M, np.int32), np.empty(M, np.int32)
    mi = np.empty(1, np.float64)
    for k in (1, 3, 5):
        for v in range(12):
            if alg == 1:
                ndf_mod.ndf_ksg_debug_pair(ctx, fid, fid, 11, v, k, a, nx, ny, mi)
                exact = H[k - 1] + H[M - 1] - sum(H[n] for c in (nx, ny) for n in map(int, c)) / M
            else:
                ndf_mod.ndf_ksg2_debug_pair(ctx, fid, fid, 11, v, k, a, b, nx, ny, mi)
                exact = (H[k - 1] - Decimal(1) / k + H[M - 1] -
                         sum(H[n - 1] for c in (nx, ny) for n in map(int, c)) / M)
            assert abs(Decimal(float(mi[0])) - exact) <= bound, (k, v, float(mi[0]), exact)
    ndf_mod.ndf_free_ensemble(ctx, fid)
