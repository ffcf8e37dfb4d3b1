"""The continuous sampler on grids whose rows start at every alignment (paired 16-byte reads of the
x-neighbours where the vertex count is a multiple of four, single reads otherwise; one-vertex axes):
positions equal to the documented SplitMix64 sequence bit for bit, KSG targets within
1e-6 |MI| + 1e-9 of the oracle on its own interpolated columns (equal columns give equal counts)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def positions(n, seed):
    def mix(z):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xbf58476d1ce4e5b9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94d049bb133111eb)
        return z ^ (z >> np.uint64(31))

    with np.errstate(over="ignore"):
        key = mix(np.array([seed], np.uint64) ^ np.uint64(0x434f4e54504f5353))
        h = mix(key + np.arange(1, 6 * n + 1, dtype=np.uint64) * np.uint64(0x9e3779b97f4a7c15)) >> np.uint64(40)
    p = (h.astype(np.float64) * (2.0 / 16777216.0) - 1.0).astype(np.float32).reshape(n, 6)
    return p[:, :3], p[:, 3:]


@pytest.mark.parametrize("X,Y,Z", [(8, 4, 2), (6, 2, 1), (1, 4, 3), (2, 2, 1), (5, 4, 1), (7, 4, 3), (3, 3, 3),
                                   (1, 1, 4), (13, 11, 3)])
def test_targets_on_ragged_grids(ndf_mod, ctx, X, Y, Z):
    M, n, k = 40, 300, 3
    f = np.random.default_rng(X * 100 + Y * 10 + Z).normal(size=(M, Z, Y, X)).astype(np.float32)
    fid = ndf_mod.ndf_load_ensemble(ctx, f, M, Z, Y, X)
    pr, pq, t = np.empty((n, 3), np.float32), np.empty((n, 3), np.float32), np.empty(n, np.float32)
    ndf_mod.ndf_sample_triples(ctx, fid, fid, ndf_mod.NDF_MEASURE_MI_KSG, k, n, 77, pr, pq, t)
    want = positions(n, 77)
    np.testing.assert_array_equal(pr, want[0])
    np.testing.assert_array_equal(pq, want[1])
    for i in range(n):
        mi = oracle.ksg_pair(oracle.interp_column(f, pr[i]), oracle.interp_column(f, pq[i]), k)[0]
        assert abs(t[i] - mi) <= 1e-6 * abs(mi) + 1e-9, (i, t[i], mi)
    ndf_mod.ndf_free_ensemble(ctx, fid)


@pytest.mark.parametrize("X,Y,Z,n", [(200, 164, 1, 8191), (200, 164, 1, 8192), (217, 151, 1, 9000), (8, 70, 70, 9001),
                                     (32768, 1, 1, 8200), (40, 30, 2, 9000)])
def test_positions_in_row_order(ndf_mod, ctx, X, Y, Z, n):
    """From 8192 positions and 32,768 vertices on they are interpolated in the order of their grid rows
    (here also more rows than its buckets, a single one, and sizes just outside): every target stays
    with its pair."""
    M, k = 20, 2
    f = np.random.default_rng(n).normal(size=(M, Z, Y, X)).astype(np.float32)
    g = np.random.default_rng(n + 1).normal(size=(M, Z, Y, X)).astype(np.float32)
    fa = ndf_mod.ndf_load_ensemble(ctx, f, M, Z, Y, X)
    fb = ndf_mod.ndf_load_ensemble(ctx, g, M, Z, Y, X)
    pr, pq, t = np.empty((n, 3), np.float32), np.empty((n, 3), np.float32), np.empty(n, np.float32)
    ndf_mod.ndf_sample_triples(ctx, fa, fb, ndf_mod.NDF_MEASURE_MI_KSG, k, n, 78, pr, pq, t)
    want = positions(n, 78)
    np.testing.assert_array_equal(pr, want[0])
    np.testing.assert_array_equal(pq, want[1])
    for i in [*range(0, n, 17), n - 1]:
        mi = oracle.ksg_pair(oracle.interp_column(f, pr[i]), oracle.interp_column(g, pq[i]), k)[0]
        assert abs(t[i] - mi) <= 1e-6 * abs(mi) + 1e-9, (i, t[i], mi)
    ndf_mod.ndf_free_ensemble(ctx, fa)
    ndf_mod.ndf_free_ensemble(ctx, fb)
