"""The dense-grid decoder where it can go wrong: grids around its 128-vertex tiles and two slots,
1 to 66 references (more than one launch), each volume bit-equal to the reference's own call and
within the BF16 bound (3e-2) of the FP64 oracle; and its biases, which are not
rounded to BF16: with zero weights the third layer is ReLU(b3) exactly, so the output is
tanh(w4 . bf16(ReLU(b3)) + b4) up to the FP32 sum over 128 terms (each bias is reproduced to 2^-24 of
itself and none of the drawn ones lies that close to a BF16 rounding boundary; 128 products of at most
0.7 in FP32: 128 * 2^-24 * 0.7 < 6e-6, bound 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_ndf import RES_SMALL, groups, make_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("X,Y,Z,R", [(1, 1, 1, 1), (127, 1, 1, 2), (128, 1, 1, 1), (43, 3, 1, 3), (16, 16, 1, 5),
                                     (257, 1, 1, 66), (131, 7, 2, 4)])
def test_tiles_and_references(ndf_mod, ctx, X, Y, Z, R):
    N = X * Y * Z
    m = ndf_mod.ndf_model_create(ctx, RES_SMALL, 0, 2, X, Y, Z)
    p = make_params(X + R)
    ndf_mod.ndf_model_set_params(m, p)
    refs = [int(v) for v in np.random.default_rng(R).integers(0, N, R)]
    out = torch.full((R, N), 9.0, device="cuda")
    torch.cuda.synchronize()
    ndf_mod.ndf_infer_batch(m, refs, out)
    ndf_mod.ndf_synchronize(ctx)  # a device output is ready on the context's stream only
    got = out.cpu().numpy()
    v = np.arange(N)
    axis = lambda i, n: -1 + 2 * i / (n - 1) if n > 1 else 0.0 * i
    pos = np.stack([axis(v % X, X), axis((v // X) % Y, Y), axis(v // (X * Y), Z)], axis=1)
    shape = oracle.net_shape(RES_SMALL, 16, 128, 0)
    for i in sorted({0, 1 % R, R // 2, R - 1}):
        one = np.empty(N, np.float32)
        ndf_mod.ndf_infer(m, refs[i], one)
        np.testing.assert_array_equal(got[i], one)
        want = oracle.ndf_forward(shape, p.astype(np.float64), np.repeat(pos[refs[i]:refs[i] + 1], N, 0), pos)
        assert np.abs(got[i] - want).max() <= 3e-2
    ndf_mod.ndf_model_free(m)


def bf16(x):
    u = x.astype(np.float32).view(np.uint32).astype(np.uint64)
    return ((u + 0x7fff + ((u >> 16) & 1)) & 0xffff0000).astype(np.uint32).view(np.float32)


def test_biases_carry_24_bits(ndf_mod, ctx):
    g, total = groups(RES_SMALL)
    rng = np.random.default_rng(3)
    p = make_params(1)
    for w in ("W1", "W2", "W3"):
        p[g[w]] = 0.0
    b3 = (rng.normal(0, 1, 128) * 10.0 ** rng.uniform(-3, 0.5, 128)).astype(np.float32)
    mid = (b3.view(np.uint32) & 0xffff).astype(np.int64) - 0x8000  # distance to a rounding boundary, in FP32 ulps
    b3[np.abs(mid) < 8] = 0.25
    p[g["b3"]] = b3
    p[g["w4"]] = rng.uniform(-0.05, 0.05, 128)
    m = ndf_mod.ndf_model_create(ctx, RES_SMALL, 0, 2, 9, 5, 3)
    ndf_mod.ndf_model_set_params(m, p)
    out = np.empty(135, np.float32)
    ndf_mod.ndf_infer(m, 7, out)
    h = bf16(np.maximum(b3, 0)).astype(np.float64)
    want = np.tanh(p[g["w4"]].astype(np.float64) @ h + float(p[g["b4"]][0]))
    assert np.abs(out - want).max() <= 1e-5
    ndf_mod.ndf_model_free(m)


def test_constant_memory_slots(ndf_mod, ctx):
    """More live models than constant-memory slots, on a grid large enough for them: every model
    decodes its own parameters, also after an update of one of them and after a slot's reuse, and a
    volume equals the one decoded in small calls (below the constant path's size)."""
    X, Y, Z = 50, 50, 20

    def make(seed):
        m = ndf_mod.ndf_model_create(ctx, RES_SMALL, 0, 2, X, Y, Z)
        ndf_mod.ndf_model_set_params(m, make_params(seed))
        return m

    def volumes(m):
        out = torch.empty((2, X * Y * Z), device="cuda")
        torch.cuda.synchronize()
        ndf_mod.ndf_infer_batch(m, [3, 777], out)
        ndf_mod.ndf_synchronize(ctx)
        one = np.empty(X * Y * Z, np.float32)
        ndf_mod.ndf_infer(m, 3, one)
        got = out.cpu().numpy()
        np.testing.assert_array_equal(got[0], one)
        return got

    models = [make(k) for k in range(20)]
    first = [volumes(m) for m in models]
    for a, b in zip(first, first[1:]):
        assert np.abs(a - b).max() > 0.05
    ndf_mod.ndf_model_set_params(models[2], make_params(99))
    changed = volumes(models[2])
    assert np.abs(changed - first[2]).max() > 0.05
    ndf_mod.ndf_model_free(models.pop(1))
    models.append(make(99))
    np.testing.assert_array_equal(volumes(models[-1]), changed)
    np.testing.assert_array_equal(volumes(models[0]), first[0])
    np.testing.assert_array_equal(volumes(models[-2]), first[19])
    for m in models:
        ndf_mod.ndf_model_free(m)


def test_constant_memory_on_two_streams(ndf_mod, ctx):
    """The first decode after an update fills the model's constant memory on its own stream; the next
    one, on another stream that does not wait for the first, reads the same values."""
    X, Y, Z = 50, 50, 20
    m = ndf_mod.ndf_model_create(ctx, RES_SMALL, 0, 2, X, Y, Z)
    ndf_mod.ndf_model_set_params(m, make_params(5))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = torch.zeros((2, 2, X * Y * Z), device="cuda")
    torch.cuda.synchronize()
    try:
        with torch.cuda.stream(streams[0]):
            torch.cuda._sleep(20_000_000)
        for s, o in zip(streams, out):
            ndf_mod.ndf_set_stream(ctx, s.cuda_stream)
            ndf_mod.ndf_infer_batch(m, [3, 777], o)
        torch.cuda.synchronize()
    finally:
        ndf_mod.ndf_set_stream(ctx, None)
    np.testing.assert_array_equal(out[1].cpu().numpy(), out[0].cpu().numpy())
    one = np.empty(X * Y * Z, np.float32)
    ndf_mod.ndf_infer(m, 3, one)
    np.testing.assert_array_equal(out[1, 0].cpu().numpy(), one)
    ndf_mod.ndf_model_free(m)
