"""One context per host thread on the same GPU: two threads whose launches of one kernel need
different amounts of shared memory (a full grid beside a handful of vertices; many references beside
few) both get every one of their calls through, with the results of calls made alone, bit for bit."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CALLS = 10000


def calls(ndf, kind, algorithm, M, N, R):
    """A thread's context and field, and one call on them: returns (call, the call with its result, close)."""
    stream = torch.cuda.Stream()
    c = ndf.ndf_create(0, stream.cuda_stream)
    f = np.random.default_rng(M + N).normal(size=(M, 1, 1, N)).astype(np.float32)
    fid = ndf.ndf_load_ensemble(c, f, M, 1, 1, N)
    out = torch.empty((R, N), device="cuda")
    if kind == "ksg":
        ndf.ndf_set_ksg_algorithm(c, getattr(ndf, algorithm))
        call = lambda: ndf.ndf_mi_ksg(c, fid, fid, N // 2, 4, out)
    else:
        refs = [i % N for i in range(R)]
        call = lambda: ndf.ndf_pearson_batch(c, fid, fid, refs, ndf.NDF_PREC_BF16X3, out)

    def once():
        call()
        ndf.ndf_synchronize(c)
        return out.cpu()

    return call, once, lambda: ndf.ndf_destroy(c)


@pytest.mark.parametrize("kind,algorithm,sizes", [
    ("ksg", "NDF_KSG_LANES", ((200, 2000, 1), (200, 5, 1))),
    ("ksg", "NDF_KSG_LANES", ((300, 2000, 1), (300, 400, 1))),
    ("ksg", "NDF_KSG_BLOCK", ((200, 2000, 1), (40, 2000, 1))),
    ("ksg", "NDF_KSG_PRUNED", ((200, 2000, 1), (40, 2000, 1))),
    ("pearson-batch", None, ((100, 1000, 64), (100, 1000, 3)))])
def test_two_threads_share_a_kernel(ndf_mod, kind, algorithm, sizes):
    users = [calls(ndf_mod, kind, algorithm, *s) for s in sizes]
    alone = [once() for _, once, _ in users]
    start = threading.Barrier(len(users))
    errors = []

    def work(call):
        start.wait()
        for i in range(CALLS):
            try:
                call()
            except Exception as e:  # noqa: BLE001 (reported by the main thread)
                errors.append((i, str(e)))
                return

    threads = [threading.Thread(target=work, args=(u[0],)) for u in users]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    after = [once() for _, once, _ in users]
    for _, _, close in users:
        close()
    assert not errors, errors
    for a, b in zip(alone, after):
        assert torch.equal(a, b)
