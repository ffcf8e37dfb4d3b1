"""The hash network's dense layers at the edges of their tiles (64 rows, 128 columns, 16-deep slices,
128-row chunks of the weight gradients; widths that are no multiple of four) against the FP64 oracle
with the bounds of test_gpu_hash (forward 2e-5 + 2e-5 |y|; gradient 1e-3 of its norm); and the
gradient returned into host memory, an aligned device buffer (which then is the step's own) and a
shifted one: the parts without atomics bit-equal, the atomically scattered grid within 1e-5 of its
norm (FP32 sums in another order), the updated parameters alike, and nothing written past the end."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_hash import HE_SCALE, archs, oshape, rand_params
from test_gpu_ndf import RES_SMALL, batch, make_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,width,merge,cross", [(1, 16, 0, False), (31, 7, 0, True), (32, 128, 0, False),
                                                 (33, 130, 3, False), (64, 20, 1, True), (65, 128, 3, True),
                                                 (127, 5, 2, False), (129, 64, 0, True), (1025, 12, 0, False)])
def test_dense_layer_edges(ndf_mod, ctx, B, width, merge, cross):
    a = archs(ndf_mod, 2, merge=merge, width=width)
    m = ndf_mod.ndf_hash_model_create(ctx, a, 0, cross, 3, 8, 8, 8)
    s = oshape(a, cross, 0)
    n = oracle.hash_param_count(s)
    p = rand_params(n, B + width, scale=HE_SCALE)
    ndf_mod.ndf_hash_model_set_params(m, p)
    rng = np.random.default_rng(B)
    pr, pq = (rng.uniform(-1, 1, (B, 3)).astype(np.float32) for _ in range(2))
    y = np.empty(B, np.float32)
    ndf_mod.ndf_hash_model_forward(m, pr, pq, y)
    ref = oracle.hash_forward(s, p.astype(np.float64), pr, pq)
    assert (np.abs(y - ref) <= 2e-5 + 2e-5 * np.abs(ref)).all()
    t = (ref + np.where(rng.uniform(size=B) < 0.5, -0.5, 0.5)).astype(np.float32)  # no sign near zero
    g = np.empty(n, np.float32)
    ndf_mod.ndf_hash_model_step(m, pr, pq, t, 0.0, False, g)
    _, gref = oracle.hash_loss_grad(s, p.astype(np.float64), pr, pq, t)
    assert np.linalg.norm(g - gref) <= 1e-3 * np.linalg.norm(gref) + 1e-7
    ndf_mod.ndf_hash_model_free(m)


@pytest.mark.parametrize("kind", ["hash", "dense"])
def test_gradient_buffers(ndf_mod, ctx, kind):
    rng = np.random.default_rng(5)
    B = 500
    pr, pq = batch(B, 3)
    t = rng.uniform(-0.9, 0.9, B).astype(np.float32)
    if kind == "hash":
        a = archs(ndf_mod, 2)
        n = oracle.hash_param_count(oshape(a, False, 0))
        p = rand_params(n, 8, scale=HE_SCALE)
        scattered = 2 * sum(min((a.base_res << l) ** 3, 1 << a.log2_table) for l in range(a.levels))
        create = lambda: ndf_mod.ndf_hash_model_create(ctx, a, 0, False, 3, 8, 8, 8)
        free, step = ndf_mod.ndf_hash_model_free, ndf_mod.ndf_hash_model_step
        put, get = ndf_mod.ndf_hash_model_set_params, ndf_mod.ndf_hash_model_get_params
    else:
        p = make_params(8)
        n, scattered = p.size, sum(r ** 3 for r in RES_SMALL) * 16
        create = lambda: ndf_mod.ndf_model_create(ctx, RES_SMALL, 0, 1, 8, 8, 8)
        free, step = ndf_mod.ndf_model_free, ndf_mod.ndf_model_step
        put, get = ndf_mod.ndf_model_set_params, ndf_mod.ndf_model_get_params
    results = []
    for shift in (None, 0, 1):  # host memory; device, 16-byte aligned; device, shifted by one float
        m = create()
        put(m, p)
        if shift is None:
            g = np.full(n, np.nan, np.float32)
            step(m, pr, pq, t, 1e-3, True, g)
        else:
            dev = torch.full((n + 8,), 7.0, device="cuda")
            torch.cuda.synchronize()
            step(m, pr, pq, t, 1e-3, True, dev[shift:shift + n])
            host = dev.cpu().numpy()
            assert (host[:shift] == 7.0).all() and (host[shift + n:] == 7.0).all()
            g = host[shift:shift + n].copy()
        step(m, pr, pq, t, 1e-3, True)  # the next step starts from a zero gradient
        after = np.empty(n, np.float32)
        get(m, after)
        results.append((g, after))
        free(m)
    g0, a0 = results[0]
    for g, after in results[1:]:
        np.testing.assert_array_equal(g[scattered:], g0[scattered:])
        assert np.linalg.norm(g[:scattered] - g0[:scattered]) <= 1e-5 * np.linalg.norm(g0[:scattered])
        # Adam's step is at most lr; gradients whose sign hangs on the atomics' order may differ
        assert np.mean(np.abs(after - a0) > 1e-5) <= 1e-3
