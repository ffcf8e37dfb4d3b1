"""The continuous sampler where it interpolates positions in the order of their grid rows: from 4,000,000
column values on (positions times members; 8,000,000 on grids of fewer than 32,768 vertices), just
below and above, with more rows than its buckets, a single row, and a second chunk that is not
ordered; and small grids of every alignment at 1000 positions and more, whose x-neighbours are read in pairs.  Positions equal the documented sequence bit for bit; KSG targets of a sample of the pairs lie
within 1e-6 |MI| + 1e-9 of the oracle on its own interpolated columns (equal columns give equal counts)."""
import numpy as np
import pytest

import oracle
from test_gpu_sampler_grids import positions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("X,Y,Z,M,n", [(200, 164, 1, 500, 7999), (200, 164, 1, 500, 8000), (8, 70, 70, 450, 9001),
                                       (32768, 1, 1, 500, 8200), (40, 30, 2, 800, 9999), (40, 30, 2, 800, 10000),
                                       (217, 151, 1, 62, 65736), (40, 30, 2, 40, 999), (40, 30, 2, 40, 1000),
                                       (7, 4, 3, 40, 1003), (1, 4, 3, 40, 1000), (2, 2, 1, 40, 1001), (13, 11, 3, 40, 1000)])
def test_targets_in_row_order(ndf_mod, ctx, X, Y, Z, M, n):
    k = 3
    rng = np.random.default_rng(n)
    f, g = (rng.normal(size=(M, Z, Y, X)).astype(np.float32) for _ in range(2))
    fa = ndf_mod.ndf_load_ensemble(ctx, f, M, Z, Y, X)
    fb = ndf_mod.ndf_load_ensemble(ctx, g, M, Z, Y, X)
    pr, pq, t = np.empty((n, 3), np.float32), np.empty((n, 3), np.float32), np.empty(n, np.float32)
    ndf_mod.ndf_sample_triples(ctx, fa, fb, ndf_mod.NDF_MEASURE_MI_KSG, k, n, 79, pr, pq, t)
    want = positions(n, 79)
    np.testing.assert_array_equal(pr, want[0])
    np.testing.assert_array_equal(pq, want[1])
    for i in [*range(0, n, n // 60), n - 150, n - 1]:
        mi = oracle.ksg_pair(oracle.interp_column(f, pr[i]), oracle.interp_column(g, pq[i]), k)[0]
        assert abs(t[i] - mi) <= 1e-6 * abs(mi) + 1e-9, (i, t[i], mi)
    ndf_mod.ndf_free_ensemble(ctx, fa)
    ndf_mod.ndf_free_ensemble(ctx, fb)
