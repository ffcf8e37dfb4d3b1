"""The default KSG search where its blocks change width: 32 to 64 x-ranks at 224 members and 64 to 128 at
850 (single pairs against the CPU oracle, bit for bit), and 256 ranks where a grid of many vertices
then fits more pairs on a SM at once (volumes against the oracle on one vertex of each kind of
column, and against the brute-force search everywhere: algorithm 1 within 1e-6 |MI| + 1e-9, FP32
output; algorithm 2 against the x-strip search alike)."""
import numpy as np
import pytest

import oracle
from test_gpu_exact import check_pairs_bit_exact, load, mi_close
from test_gpu_ksg_lanes import mixed_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,k", [(223, 4), (224, 8), (225, 8), (850, 8), (851, 8)])
def test_block_width_edges(ndf_mod, ctx, M, k):
    f = mixed_field(M, M)
    fid = load(ndf_mod, ctx, f)
    for r in (0, 1, 3):
        check_pairs_bit_exact(ndf_mod, ctx, fid, fid, f, f, r, range(f[0].size), k)
    ndf_mod.ndf_free_ensemble(ctx, fid)


@pytest.mark.parametrize("M,N", [(1100, 1750), (1701, 1000), (1800, 1100), (2049, 2000), (2500, 700), (3000, 500),
                                 (4096, 700)])
def test_wide_blocks(ndf_mod, ctx, M, N):
    few = mixed_field(M, M).reshape(M, 10)
    many = np.random.default_rng(M).normal(size=(M, N)).astype(np.float32)
    many += 0.7 * few[:, :1]
    many[:, :10] = few
    many[:, N - 10:] = few
    f = np.ascontiguousarray(many.reshape(M, 1, 1, N))
    fid = load(ndf_mod, ctx, f)
    columns = np.ascontiguousarray(f[..., :10])
    for k in (3, 8):
        for r in (0, 1):
            out, brute = np.empty(N, np.float32), np.empty(N, np.float32)
            ndf_mod.ndf_mi_ksg(ctx, fid, fid, r, k, out)
            ndf_mod.ndf_set_ksg_algorithm(ctx, ndf_mod.NDF_KSG_BRUTE)
            ndf_mod.ndf_mi_ksg(ctx, fid, fid, r, k, brute)
            ndf_mod.ndf_set_ksg_algorithm(ctx, ndf_mod.NDF_KSG_LANES)
            ok, where = mi_close(out, brute.astype(np.float64))
            assert ok, (k, r, where)
            np.testing.assert_array_equal(out[:10], out[N - 10:])
            ok, where = mi_close(out[:10].reshape(1, 1, 10), oracle.ksg_volume(columns, columns, r, k))
            assert ok, (k, r, where)
            ndf_mod.ndf_mi_ksg2(ctx, fid, fid, r, k, out)
            ndf_mod.ndf_set_ksg_algorithm(ctx, ndf_mod.NDF_KSG_PRUNED)
            ndf_mod.ndf_mi_ksg2(ctx, fid, fid, r, k, brute)
            ndf_mod.ndf_set_ksg_algorithm(ctx, ndf_mod.NDF_KSG_LANES)
            ok, where = mi_close(out, brute.astype(np.float64))
            assert ok, (k, r, where)
    batch = np.empty((2, N), np.float32)
    ndf_mod.ndf_mi_ksg_batch(ctx, fid, fid, [0, 1], 8, batch)
    ndf_mod.ndf_mi_ksg(ctx, fid, fid, 1, 8, brute)
    np.testing.assert_array_equal(batch[1], brute)
    ndf_mod.ndf_free_ensemble(ctx, fid)
