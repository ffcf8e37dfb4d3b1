"""Device memory of the hash network's calls follows what they do: a forward call or an FP32 decode
takes no room for gradient sums, and a step's follow its batch (a batch of up to 128 pairs one set of
sums).  Limits: the activations of the batch (two buffers of both sides' rows per layer and eight more, each
of the widest layer) and, for a step, the sums of every layer; 8 MB more for the allocator's granularity."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("width,cross,B", [(1024, True, 1), (1024, False, 100), (128, False, 1), (256, True, 300)])
def test_call_memory(ndf_mod, ctx, width, cross, B):
    a = ndf_mod.ndf_hash_arch_default()
    a.width, a.log2_table = width, 10
    rng = np.random.default_rng(0)
    pr, pq = (rng.uniform(-1, 1, (B, 3)).astype(np.float32) for _ in range(2))
    y = np.empty(B, np.float32)
    out = torch.empty(4 * 4 * 2, device="cuda")
    small = ndf_mod.ndf_hash_arch_default()
    small.width, small.log2_table = 8, 4
    warm = ndf_mod.ndf_hash_model_create(ctx, small, 0, cross, 3, 4, 4, 2)  # loads the kernels
    ndf_mod.ndf_hash_set_decode(warm, ndf_mod.NDF_HASH_DECODE_FP32)
    ndf_mod.ndf_hash_infer(warm, 3, out)
    ndf_mod.ndf_hash_model_step(warm, pr[:1], pq[:1], np.zeros(1, np.float32), 0.0, False)
    ndf_mod.ndf_hash_model_free(warm)
    m = ndf_mod.ndf_hash_model_create(ctx, a, 0, cross, 3, 4, 4, 2)
    ndf_mod.ndf_hash_set_decode(m, ndf_mod.NDF_HASH_DECODE_FP32)
    layers = a.enc_layers + a.dec_layers
    wide = max(width, 3 + 6 * a.n_freq + a.levels * a.feat)
    rows = 2 * max(B, 32)  # the decode's batch is the grid's 32 vertices
    activations = 4 * rows * wide * (2 * layers + 8) + (8 << 20)
    sets = (2 if cross else 1) * a.enc_layers * -(-(B if cross else 2 * B) // 128) + a.dec_layers * -(-B // 128)
    sums = 4 * sets * wide * (wide + 1) + (8 << 20)
    before = free_bytes()
    ndf_mod.ndf_hash_model_forward(m, pr, pq, y)
    ndf_mod.ndf_hash_infer(m, 3, out)
    forward = before - free_bytes()
    assert forward <= activations, (forward, activations)
    before = free_bytes()
    ndf_mod.ndf_hash_model_step(m, pr, pq, y, 0.0, False)
    step = before - free_bytes()
    assert step <= sums, (step, sums)
    ndf_mod.ndf_hash_model_free(m)
