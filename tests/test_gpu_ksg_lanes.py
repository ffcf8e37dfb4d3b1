"""The default KSG search at the edges of its block sizes (32, 64 and 128 x-ranks by M), on columns
with ties, half of them equal, or all equal, and the staging of the reference columns (one warp per
reference for few members or many references, one CTA otherwise): eps and counts bit-exact against
the CPU oracle, MI within 1e-6 |MI| + 1e-9 (FP32 output), batched volumes equal to single ones bit for
bit."""
import numpy as np
import pytest

import oracle
from test_gpu_exact import check_pairs_bit_exact, load, mi_close

pytestmark = pytest.mark.gpu


def mixed_field(M, seed):
    """Columns: normal, rounded to 1/4, half zeros, constant, constant but one member, +-0."""
    f = np.random.default_rng(seed).normal(size=(M, 1, 2, 5)).astype(np.float32)
    f[:, 0, 0, 1] = np.round(f[:, 0, 0, 1] * 4) / 4
    f[:, 0, 0, 2] = np.maximum(f[:, 0, 0, 2], 0)
    f[:, 0, 0, 3] = 1.5
    f[:, 0, 0, 4] = -2.0
    f[M // 2, 0, 0, 4] = 3.0
    f[:, 0, 1, 0] = np.where(np.arange(M) % 2 == 0, np.float32(-0.0), np.float32(0.0))
    return f


@pytest.mark.parametrize("M,k", [(31, 3), (32, 4), (33, 5), (64, 4), (65, 4), (128, 5), (129, 5), (255, 6), (256, 6),
                                 (257, 6), (512, 8), (513, 8), (768, 8), (769, 8), (1000, 12), (1025, 8), (2049, 3)])
def test_lane_search_block_edges(ndf_mod, ctx, M, k):
    f = mixed_field(M, M)
    fid = load(ndf_mod, ctx, f)
    N = f[0].size
    for r in (0, 1, 3):  # a normal, a tied and a constant reference
        check_pairs_bit_exact(ndf_mod, ctx, fid, fid, f, f, r, range(N), k)
        out = np.empty(N, np.float32)
        ndf_mod.ndf_mi_ksg(ctx, fid, fid, r, k, out)
        ok, where = mi_close(out, oracle.ksg_volume(f, f, r, k))
        assert ok, (r, where)
    ndf_mod.ndf_free_ensemble(ctx, fid)


@pytest.mark.parametrize("M,R", [(100, 3), (128, 5), (129, 1), (256, 7), (257, 32), (300, 33), (512, 40), (513, 32),
                                 (1000, 37), (1024, 32), (1025, 33)])
def test_staged_references_match_single_calls(ndf_mod, ctx, M, R):
    f = mixed_field(M, 7 * M)
    fid = load(ndf_mod, ctx, f)
    N = f[0].size
    refs = [i % N for i in range(R)]
    out = np.empty((R, N), np.float32)
    ndf_mod.ndf_mi_ksg_batch(ctx, fid, fid, refs, 4, out)
    one = np.empty(N, np.float32)
    for r in range(min(R, N)):
        ndf_mod.ndf_mi_ksg(ctx, fid, fid, r, 4, one)
        rows = out[r::N]
        np.testing.assert_array_equal(rows, np.broadcast_to(one, rows.shape))
        ok, where = mi_close(one, oracle.ksg_volume(f, f, r, 4))
        assert ok, (r, where)
    ndf_mod.ndf_free_ensemble(ctx, fid)
