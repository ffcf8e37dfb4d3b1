"""Training steps of the hash network at the limits of its gradient sums, against the FP64 oracle with
the bound of test_gpu_hash (1e-3 of the gradient's norm): batches of which a CTA of the output layer takes
several groups of rows and the layers the most chunks of rows (8193, 20,001: the last ones short), and
networks whose sums do not all fit their workspace or their list, which are then added in the middle of a step
(width 1024; two encoders of eight layers).  The parts without atomics are bit-equal in a second step,
and in a model that has seen other inputs and batch sizes before: nothing is read before it is written."""
import numpy as np
import pytest

import oracle
from test_gpu_hash import archs, oshape, rand_params

pytestmark = pytest.mark.gpu


def inputs(B, seed):
    rng = np.random.default_rng(seed)
    pr, pq = (rng.uniform(-1, 1, (B, 3)).astype(np.float32) for _ in range(2))
    return pr, pq, np.where(rng.uniform(size=B) < 0.5, -0.5, 0.5)


def dense_part(a, cross, n):
    """Mask of the parameters outside the hash tables."""
    tables = a.feat * sum(min((a.base_res << l) ** 3, 1 << a.log2_table) for l in range(a.levels))
    din = 3 + 6 * a.n_freq + a.levels * a.feat
    encoder = tables + a.enc_layers * a.width + sum((din if k == 0 else a.width) * a.width
                                                    for k in range(a.enc_layers))
    mask = np.ones(n, bool)
    for e in range(2 if cross else 1):
        mask[e * encoder:e * encoder + tables] = False
    return mask


@pytest.mark.parametrize("B,cross,kw", [(8193, False, dict(width=12)), (20001, False, dict(width=12)),
                                        (20001, True, dict(width=20, merge=3)),
                                        (129, False, dict(width=1024, enc_layers=8, dec_layers=8)),
                                        (100, True, dict(width=16, enc_layers=8, dec_layers=5))])
def test_gradients_at_the_limits(ndf_mod, ctx, B, cross, kw):
    a = archs(ndf_mod, 2, **kw)
    m = ndf_mod.ndf_hash_model_create(ctx, a, 0, cross, 3, 8, 8, 8)
    s = oshape(a, cross, 0)
    n = oracle.hash_param_count(s)
    p = rand_params(n, B, scale=(2.0 / a.width) ** 0.5)
    ndf_mod.ndf_hash_model_set_params(m, p)
    pr, pq, off = inputs(B, B)
    y = np.empty(B, np.float32)
    ndf_mod.ndf_hash_model_forward(m, pr, pq, y)
    t = (y + off).astype(np.float32)  # no sign near zero
    g, again = np.empty(n, np.float32), np.empty(n, np.float32)
    ndf_mod.ndf_hash_model_step(m, pr, pq, t, 0.0, False, g)
    _, gref = oracle.hash_loss_grad(s, p.astype(np.float64), pr, pq, t)
    assert np.linalg.norm(g - gref) <= 1e-3 * np.linalg.norm(gref) + 1e-7
    dense = dense_part(a, cross, n)
    assert np.linalg.norm((g - gref)[dense]) <= 1e-3 * np.linalg.norm(gref[dense]) + 1e-7
    ndf_mod.ndf_hash_model_step(m, pr, pq, t, 0.0, False, again)
    np.testing.assert_array_equal(again[dense], g[dense])
    ndf_mod.ndf_hash_model_free(m)


@pytest.mark.parametrize("cross,kw", [(False, dict(width=128, enc_layers=6, dec_layers=6)), (True, dict(width=64)),
                                      (False, dict(width=32, enc_layers=0))])
def test_steps_after_other_inputs(ndf_mod, ctx, cross, kw):
    a = archs(ndf_mod, 2, **kw)
    n = oracle.hash_param_count(oshape(a, cross, 0))
    p = rand_params(n, 5, scale=(2.0 / a.width) ** 0.5)
    dense = dense_part(a, cross, n)
    for B in (8192, 3000, 37):
        pr, pq, t = inputs(B, B)
        t = t.astype(np.float32)
        results = []
        for before in ((), (20000, 5, 8192, 700, B)):
            m = ndf_mod.ndf_hash_model_create(ctx, a, 0, cross, 3, 8, 8, 8)
            ndf_mod.ndf_hash_model_set_params(m, p)
            for i, b in enumerate(before):
                qr, qq, u = inputs(b, 100 + i)
                ndf_mod.ndf_hash_model_step(m, qr, qq, u.astype(np.float32), 0.0, False)
                ndf_mod.ndf_hash_model_forward(m, qq, qr, np.empty(b, np.float32))
            g = np.empty(n, np.float32)
            loss = ndf_mod.ndf_hash_model_step(m, pr, pq, t, 0.0, False, g)
            results.append((loss, g))
            ndf_mod.ndf_hash_model_free(m)
        (l0, g0), (l1, g1) = results
        assert l1 == pytest.approx(l0, rel=1e-12)
        np.testing.assert_array_equal(g1[dense], g0[dense])
        assert np.linalg.norm((g1 - g0)[~dense]) <= 1e-5 * np.linalg.norm(g0[~dense])
