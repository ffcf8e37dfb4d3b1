"""A dense-network decode captured in a CUDA graph (which reads the biases from the parameters, not from the
constant-memory copy): replays follow parameter updates and equal ordinary decodes bit for bit."""
import numpy as np
import pytest
import torch

from test_gpu_ndf import RES_SMALL, make_params

pytestmark = pytest.mark.gpu


def test_captured_decode_follows_updates(ndf_mod, ctx):
    X, Y, Z = 50, 50, 20
    m = ndf_mod.ndf_model_create(ctx, RES_SMALL, 0, 2, X, Y, Z)
    ndf_mod.ndf_model_set_params(m, make_params(5))
    refs = np.array([3, 777], np.int64)  # read by every replay
    out = torch.zeros((2, X * Y * Z), device="cuda")
    want = torch.zeros_like(out)
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    try:
        ndf_mod.ndf_set_stream(ctx, stream.cuda_stream)
        ndf_mod.ndf_infer_batch(m, refs, want)  # sizes the scratch
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            ndf_mod.ndf_infer_batch(m, refs, out)
        for seed in (5, 6, 7):
            ndf_mod.ndf_model_set_params(m, make_params(seed))
            ndf_mod.ndf_infer_batch(m, refs, want)
            ndf_mod.ndf_synchronize(ctx)
            out.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, want), seed
    finally:
        ndf_mod.ndf_set_stream(ctx, None)
        ndf_mod.ndf_model_free(m)
