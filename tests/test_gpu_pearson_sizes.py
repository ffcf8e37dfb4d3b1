"""A Pearson volume takes one of three kernels by its vertex count (one launch with one or four
vertices per thread, or staged reference and volume): at the edges of their ranges, and for member
counts around their row batches, every vertex's value is the same bits whichever kernel its grid
takes (slabs of a grid equal the grid), and within 1e-5 of the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [2, 15, 63, 64, 65, 129])
def test_same_bits_at_every_size(ndf_mod, ctx, M):
    big = 262148  # above the one-launch range
    f = torch.randn((M, big), generator=torch.Generator(device="cuda").manual_seed(M), device="cuda")
    f[:, 3] = 2.5
    torch.cuda.synchronize()
    ref = 11
    whole = ndf_mod.ndf_load_ensemble(ctx, f, M, 1, 1, big)
    want = np.empty(big, np.float32)
    ndf_mod.ndf_pearson(ctx, whole, whole, ref, want)
    ndf_mod.ndf_free_ensemble(ctx, whole)
    col = f[:, ref].cpu().numpy().copy()
    for n in (1, 3, 12, 127, 128, 129, 513, 65535, 65536, 65537, 65540, 262144):
        part = f[:, :n].contiguous()
        torch.cuda.synchronize()
        fid = ndf_mod.ndf_load_ensemble(ctx, part, M, 1, 1, n)
        out = np.empty(n, np.float32)
        ndf_mod.ndf_pearson_column(ctx, col, fid, out)
        np.testing.assert_array_equal(out, want[:n], err_msg=str(n))
        if n > ref:
            ndf_mod.ndf_pearson(ctx, fid, fid, ref, out)
            np.testing.assert_array_equal(out, want[:n], err_msg=str(n))
        if n == 129:
            host = part.cpu().numpy().reshape(M, 1, 1, n)
            assert np.abs(out - oracle.pearson_volume(host, host, ref)).max() <= 1e-5
        ndf_mod.ndf_free_ensemble(ctx, fid)


def test_many_members(ndf_mod, ctx):
    """The largest member counts on either side of the one-launch range."""
    for M in (8192, 8193):
        f = np.random.default_rng(M).normal(size=(M, 1, 2, 20)).astype(np.float32)
        fid = ndf_mod.ndf_load_ensemble(ctx, f, M, 1, 2, 20)
        out = np.empty(40, np.float32)
        ndf_mod.ndf_pearson(ctx, fid, fid, 7, out)
        assert np.abs(out - oracle.pearson_volume(f, f, 7).ravel()).max() <= 1e-5
        ndf_mod.ndf_free_ensemble(ctx, fid)
