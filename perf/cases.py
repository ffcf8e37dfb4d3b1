"""Performance cases: the calls a program makes on the dependence-volume library.

Every case is a dict of plain values.  ``listed()`` names the standing ones, ``draw()`` gives
further ones of the same ranges, ``prepare()`` builds what the program has in hand before the
call (ensembles on the device, loaded fields, models with their parameters), ``run()`` makes one
call through the public entry points and returns its outputs, ``exact()`` gives the outputs in
64 bits from the definitions alone, and ``work()`` the bytes and operations of one call.

Kinds:
  pearson         one reference vertex against every vertex (an interactive click)
  pearson-batch   many references at once on the tensor cores (precomputed volumes)
  ksg             KSG mutual information of one or several references against every vertex
  load            a device-resident ensemble handed to the library: copy, statistics, sorted columns
  triples         continuous training samples (positions and their dependence)
  dense-step      one Adam step of the dense-grid network, with its gradient
  dense-decode    volumes decoded by the dense-grid network
  hash-step       one Adam step of the hash-grid network (the paper's), with its gradient
  hash-decode     volumes decoded by the hash-grid network
"""
import math

import numpy as np
import torch

from paper_2307_02203_gb300 import ndf

DEVICE = "cuda"


def listed():
    return [
        # the smallest grid a user explores (16 x 16 x 4, 100 members): one click, all latency
        {"name": "pearson-tiny", "kind": "pearson", "X": 16, "Y": 16, "Z": 4, "M": 100,
         "cross": False, "packed": False},
        # the paper's grid and ensemble: one click, the whole 7 GB field streamed
        {"name": "pearson-paper-grid", "kind": "pearson", "X": 250, "Y": 352, "Z": 20, "M": 1000,
         "cross": False, "packed": False},
        # 64 references at once (correlation matrices between regions), split-BF16 products
        {"name": "pearson-batch", "kind": "pearson-batch", "X": 250, "Y": 352, "Z": 5, "M": 1000,
         "R": 64, "prec": "bf16x3"},
        # the smallest mutual-information volume: one click on the small grid
        {"name": "ksg-tiny", "kind": "ksg", "X": 16, "Y": 16, "Z": 4, "M": 100, "k": 4, "alg": 1,
         "R": 1, "cross": False, "packed": False},
        # two variables of an odd-sized region, values packed to few bits as archives store them
        {"name": "ksg-ragged-cross", "kind": "ksg", "X": 61, "Y": 43, "Z": 7, "M": 333, "k": 5,
         "alg": 1, "R": 1, "cross": True, "packed": True},
        # the paper's timed workload: one mutual-information volume of the full grid
        {"name": "ksg-paper-grid", "kind": "ksg", "X": 250, "Y": 352, "Z": 20, "M": 1000, "k": 8,
         "alg": 1, "R": 1, "cross": False, "packed": False},
        # an ensemble that a simulation left on the device is taken over for exploration
        {"name": "load-device", "kind": "load", "X": 250, "Y": 352, "Z": 4, "M": 1000},
        # training data of the mutual-information network: fresh random pairs of positions
        {"name": "triples-ksg", "kind": "triples", "X": 125, "Y": 176, "Z": 20, "M": 500, "k": 8,
         "measure": "mi", "n": 100000},
        # training of the dense-grid network at its default grid and batch
        {"name": "dense-step", "kind": "dense-step", "res": 32, "B": 1 << 18, "measure": "pearson"},
        # 16 decoded volumes of the paper's grid at once (a row of linked views)
        {"name": "dense-decode", "kind": "dense-decode", "X": 250, "Y": 352, "Z": 20, "res": 32,
         "R": 16, "measure": "pearson"},
        # training of the paper's network at its usual batch
        {"name": "hash-step", "kind": "hash-step", "B": 8192, "cross": False, "measure": "pearson",
         "act": 2, "merge": 0},
        # one decoded volume of the paper's grid by the paper's network (an interactive click)
        {"name": "hash-decode", "kind": "hash-decode", "X": 250, "Y": 352, "Z": 20, "R": 1,
         "measure": "pearson", "mode": "tc"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, n_max, n_min=600):
    """X, Y, Z of about n vertices, n log-uniform; flat like an atmosphere."""
    n = _log_int(rng, n_min, n_max)
    Z = max(1, min(20, _log_int(rng, 1, 20)))
    side = max(2.0, math.sqrt(n / Z))
    X = max(2, int(side * rng.uniform(0.7, 1.2)))
    return X, max(2, int(n / Z / X)), Z


def draw(rng):
    kind = rng.choice(["pearson", "pearson-batch", "ksg", "ksg", "load", "triples", "dense-step",
                       "dense-decode", "hash-step", "hash-step", "hash-decode"])
    c = {"kind": kind}
    if kind in ("pearson", "pearson-batch", "ksg", "load", "triples"):
        M = _log_int(rng, 60, 1800)
        n_max = {"pearson": 1760000, "pearson-batch": 440000, "ksg": 300000, "load": 350000,
                 "triples": 440000}[kind]
        c["X"], c["Y"], c["Z"] = _grid(rng, min(n_max, int(n_max * 1000 / max(M, 250))))
        c["M"] = M
    if kind == "pearson":
        c["cross"], c["packed"] = rng.random() < 0.3, rng.random() < 0.3
    elif kind == "pearson-batch":
        c["R"] = rng.randint(2, 130)
        c["prec"] = rng.choice(["bf16x3", "tf32"])
    elif kind == "ksg":
        c["k"] = rng.randint(3, 12)
        c["alg"] = 2 if rng.random() < 0.25 else 1
        c["R"] = 1 if c["alg"] == 2 else rng.choice([1, 1, 1, 3])
        c["cross"], c["packed"] = rng.random() < 0.4, rng.random() < 0.3
    elif kind == "triples":
        c["measure"] = rng.choice(["pearson", "mi"])
        c["k"] = rng.randint(3, 10)
        c["n"] = _log_int(rng, 2000, 200000)
    elif kind == "dense-step":
        c["res"] = rng.choice([8, 16, 32])
        c["B"] = _log_int(rng, 1000, 1 << 18)
        c["measure"] = rng.choice(["pearson", "mi"])
    elif kind == "dense-decode":
        c["X"], c["Y"], c["Z"] = _grid(rng, 1760000, 5000)
        c["res"] = rng.choice([16, 32])
        c["R"] = rng.randint(1, 24)
        c["measure"] = rng.choice(["pearson", "mi"])
    elif kind == "hash-step":
        c["B"] = _log_int(rng, 1000, 20000)
        c["cross"] = rng.random() < 0.3
        c["measure"] = rng.choice(["pearson", "mi"])
        c["act"] = rng.choice([1, 2, 2])
        c["merge"] = rng.choice([0, 0, 1, 3])
    elif kind == "hash-decode":
        c["mode"] = rng.choice(["tc", "tc", "cached", "fp32"])
        c["X"], c["Y"], c["Z"] = _grid(rng, 300000 if c["mode"] == "fp32" else 1760000, 5000)
        c["R"] = 1 if c["mode"] == "fp32" else rng.randint(1, 10)
        c["measure"] = rng.choice(["pearson", "mi"])
    return c


# ---------------------------------------------------------------- inputs
def _generator(seed, stream):
    g = torch.Generator(device=DEVICE)
    g.manual_seed((int(seed) * 1000003 + stream) % (1 << 62))
    return g


def _smoothing(n, sigma):
    """[n, n] matrix of a Gaussian of width sigma, unit power, reflected at the ends."""
    radius = int(math.ceil(4 * sigma))
    t = np.arange(-radius, radius + 1)
    w = np.exp(-0.5 * (t / sigma) ** 2)
    w /= math.sqrt(float((w * w).sum()))
    a = np.zeros((n, n))
    for i in range(n):
        j = (i + t) % (2 * n)
        np.add.at(a[i], np.where(j < n, j, 2 * n - 1 - j), w)
    return torch.tensor(a, dtype=torch.float32, device=DEVICE)


def _smooth_noise(M, Z, Y, X, gen):
    u = torch.randn((M, Z, Y, X), generator=gen, device=DEVICE)
    u = u @ _smoothing(X, min(12.0, X / 4)).T
    u = _smoothing(Y, min(12.0, Y / 4)) @ u
    if Z > 1:
        u = torch.einsum("zw,mwyx->mzyx", _smoothing(Z, min(3.0, Z / 3)), u)
    return u


def _transform(u, packed):
    """Skewed values on even levels, heavy tails on odd ones; packed to 1/256 steps if wanted."""
    out = u + 0.3 * u * u  # [M, Z, Y, X]
    odd = u[:, 1::2]
    out[:, 1::2] = torch.sign(odd) * odd.abs() ** 1.5
    return ((out * 256.0).round() / 256.0 if packed else out).contiguous()


def _ensembles(case, seed):
    """The member-major field(s) [M, Z, Y, X]: smooth noise, three shared modes; a second
    variable shares 0.6 of the first."""
    M, Z, Y, X = case["M"], case["Z"], case["Y"], case["X"]
    gen = _generator(seed, 1)
    u = _smooth_noise(M, Z, Y, X, gen)
    amp = torch.randn((3, M), generator=gen, device=DEVICE)
    x = torch.arange(X, device=DEVICE) / X
    y = torch.arange(Y, device=DEVICE) / Y
    for q in range(3):
        mode = torch.sin(2 * math.pi * (q + 1) * x)[None, :] * torch.cos(math.pi * q * y)[:, None]
        u += amp[q][:, None, None, None] * mode
    fields = [_transform(u, case.get("packed", False))]
    if case.get("cross"):
        fields.append(_transform(0.6 * u + 0.8 * _smooth_noise(M, Z, Y, X, gen),
                                 case.get("packed", False)))
    return fields


def _references(case, seed, count):
    n = case["X"] * case["Y"] * case["Z"]
    return [int(v) for v in np.random.RandomState(int(seed) % (1 << 31)).randint(0, n, count)]


DENSE_FEATURES, WIDTH = 16, 128


def _dense_res(case):
    return [case["res"] * (1 << i) for i in range(4)]


def _dense_params(case, seed):
    """A trained-like parameter vector: grid features of a few tenths, He-sized layers."""
    gen = _generator(seed, 2)
    n_grid = sum(r ** 3 for r in _dense_res(case)) * DENSE_FEATURES
    n_mlp = 3 * (WIDTH * WIDTH + WIDTH) + WIDTH + 1
    p = torch.empty(n_grid + n_mlp, device=DEVICE)
    p[:n_grid].uniform_(-0.3, 0.3, generator=gen)
    p[n_grid:].uniform_(-1.0, 1.0, generator=gen)
    p[n_grid:] *= math.sqrt(6.0 / WIDTH)
    o = n_grid
    for _ in range(3):
        p[o + WIDTH * WIDTH:o + WIDTH * WIDTH + WIDTH] *= 0.1
        o += WIDTH * WIDTH + WIDTH
    p[-1] = 0.1
    return p


def _hash_layout(case):
    """(levels, offsets) of the paper's network: 6 hash levels from 16^3 with 2^22 entries,
    12 Fourier frequencies, encoders and decoder of 6 x 128."""
    levels, off = [], 0
    for l in range(6):
        res = 16 << l
        entries = min(res ** 3, 1 << 22)
        levels.append((res, entries, off, res ** 3 <= 1 << 22))
        off += entries * 2
    d_in, layers = 3 + 6 * 12 + 6 * 2, []
    for k in range(6):
        c_in = d_in if k == 0 else WIDTH
        layers.append((off, off + c_in * WIDTH, c_in, WIDTH))
        off += c_in * WIDTH + WIDTH
    enc_size, n_enc = off, 2 if case.get("cross") else 1
    off = enc_size * n_enc
    d_dec, dec = (2 * WIDTH if case.get("merge", 0) == 3 else WIDTH), []
    for k in range(6):
        c_in, c_out = (d_dec if k == 0 else WIDTH), (1 if k == 5 else WIDTH)
        dec.append((off, off + c_in * c_out, c_in, c_out))
        off += c_in * c_out + c_out
    return levels, layers, dec, enc_size, n_enc, off


def _hash_params(case, seed, last):
    """An early-training parameter vector: the usual initial scales, small biases, output
    weights of U(-last, last)."""
    gen = _generator(seed, 3)
    levels, enc, dec, enc_size, n_enc, total = _hash_layout(case)
    p = torch.empty(total, device=DEVICE).uniform_(-1.0, 1.0, generator=gen)
    tables = enc[0][0]

    def layer(base, w, b, c_in, c_out, scale):
        p[base + w:base + b] *= scale
        p[base + b:base + b + c_out] *= 0.05

    for e in range(n_enc):
        base = e * enc_size
        p[base:base + tables] *= 0.1
        for k, (w, b, c_in, c_out) in enumerate(enc):
            layer(base, w, b, c_in, c_out, 0.9 * math.sqrt(6.0 / c_in))
            if k == 0:
                p[base + w:base + b].view(c_out, c_in)[:, 3:75] *= 0.1
    for k, (w, b, c_in, c_out) in enumerate(dec):
        layer(0, w, b, c_in, c_out, last if k == 5 else 0.9 * math.sqrt(6.0 / c_in))
    return p


def _batch(case, seed):
    """Positions of B pairs and targets well away from the untrained predictions: correlations
    of magnitude 0.25 to 1, or mutual information of 1 to 4 nats."""
    gen = _generator(seed, 4)
    B = case["B"]
    pr = torch.empty((B, 3), device=DEVICE).uniform_(-1.0, 1.0, generator=gen)
    pq = torch.empty((B, 3), device=DEVICE).uniform_(-1.0, 1.0, generator=gen)
    u = torch.empty(B, device=DEVICE).uniform_(-1.0, 1.0, generator=gen)
    if case["measure"] == "pearson":
        return pr, pq, torch.where(u < 0, 0.75 * u - 0.25, 0.75 * u + 0.25)
    return pr, pq, 2.5 + 1.5 * u


def _measure(case):
    return ndf.NDF_MEASURE_PEARSON if case["measure"] == "pearson" else ndf.NDF_MEASURE_MI_KSG


def _hash_arch(case):
    a = ndf.ndf_hash_arch_default()
    a.act, a.merge = case.get("act", 2), case.get("merge", 0)
    return a


class _State:
    """A program's context on its own stream, with the handles and buffers it keeps."""

    def __init__(self, case):
        self.case = case
        self.stream = torch.cuda.Stream()
        self.ctx = ndf.ndf_create(torch.cuda.current_device(), self.stream.cuda_stream)
        self.dense = self.hash = None

    def __del__(self):
        if self.dense is not None:
            ndf.ndf_model_free(self.dense)
        if self.hash is not None:
            ndf.ndf_hash_model_free(self.hash)
        ndf.ndf_destroy(self.ctx)


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind in ("pearson", "pearson-batch", "ksg", "triples", "load"):
        M, Z, Y, X = case["M"], case["Z"], case["Y"], case["X"]
        N = Z * Y * X
        fields = _ensembles(case, seed)
        torch.cuda.synchronize()
        if kind == "load":
            s.field = fields[0]
            s.mean = torch.empty(N, dtype=torch.float64, device=DEVICE)
            s.inv_norm = torch.empty(N, dtype=torch.float64, device=DEVICE)
            s.columns = torch.empty((M, N), device=DEVICE)
            return s
        ids = [ndf.ndf_load_ensemble(s.ctx, f, M, Z, Y, X) for f in fields]
        s.a, s.b = ids[0], ids[-1]
        R = case.get("R", 1)
        s.refs = _references(case, seed, R)
        if kind == "triples":
            n = case["n"]
            s.seed = int(seed)
            s.pref = torch.empty((n, 3), device=DEVICE)
            s.pq = torch.empty((n, 3), device=DEVICE)
            s.target = torch.empty(n, device=DEVICE)
        else:
            s.out = torch.empty((R, N), device=DEVICE)
        return s
    if kind.startswith("dense"):
        X, Y, Z = (case.get(a, d) for a, d in (("X", 250), ("Y", 352), ("Z", 20)))
        s.dense = ndf.ndf_model_create(s.ctx, _dense_res(case), _measure(case), 1, X, Y, Z)
        params = _dense_params(case, seed)
        assert params.numel() == ndf.ndf_model_param_count(s.dense)
        torch.cuda.synchronize()
        ndf.ndf_model_set_params(s.dense, params)
    else:
        X, Y, Z = (case.get(a, d) for a, d in (("X", 250), ("Y", 352), ("Z", 20)))
        s.hash = ndf.ndf_hash_model_create(s.ctx, _hash_arch(case), _measure(case),
                                           case.get("cross", False), 1, X, Y, Z)
        params = _hash_params(case, seed, 0.02 if kind == "hash-step" else 0.3)
        assert params.numel() == ndf.ndf_hash_model_param_count(s.hash)
        torch.cuda.synchronize()
        ndf.ndf_hash_model_set_params(s.hash, params)
        if kind == "hash-decode":
            mode = ndf.NDF_HASH_DECODE_FP32 if case["mode"] == "fp32" else ndf.NDF_HASH_DECODE_TC
            ndf.ndf_hash_set_decode(s.hash, mode, case["mode"] == "cached")
    if kind.endswith("step"):
        s.pr, s.pq, s.target = _batch(case, seed)
        s.grad = torch.empty_like(params)
    else:
        s.refs = _references(case, seed, case["R"])
        s.out = torch.empty((case["R"], X * Y * Z), device=DEVICE)
    torch.cuda.synchronize()
    return s


def _parts(case, grad):
    """A gradient by its parts, whose sizes differ by orders of magnitude."""
    if case["kind"] == "dense-step":
        n = sum(r ** 3 for r in _dense_res(case)) * DENSE_FEATURES
        return {"grid": grad[:n], "mlp": grad[n:]}
    _, enc, _, enc_size, n_enc, _ = _hash_layout(case)
    d = {"decoder": grad[enc_size * n_enc:]}
    for e in range(n_enc):
        d["tables%d" % e] = grad[e * enc_size:e * enc_size + enc[0][0]]
        d["encoder%d" % e] = grad[e * enc_size + enc[0][0]:(e + 1) * enc_size]
    return d


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "pearson":
        ndf.ndf_pearson(s.ctx, s.a, s.b, s.refs[0], s.out)
        return s.out
    if kind == "pearson-batch":
        prec = ndf.NDF_PREC_BF16X3 if case["prec"] == "bf16x3" else ndf.NDF_PREC_TF32
        ndf.ndf_pearson_batch(s.ctx, s.a, s.b, s.refs, prec, s.out)
        return s.out
    if kind == "ksg":
        if case["alg"] == 2:
            ndf.ndf_mi_ksg2(s.ctx, s.a, s.b, s.refs[0], case["k"], s.out)
        elif case["R"] == 1:
            ndf.ndf_mi_ksg(s.ctx, s.a, s.b, s.refs[0], case["k"], s.out)
        else:
            ndf.ndf_mi_ksg_batch(s.ctx, s.a, s.b, s.refs, case["k"], s.out)
        return s.out
    if kind == "load":
        fid = ndf.ndf_load_ensemble(s.ctx, s.field, case["M"], case["Z"], case["Y"], case["X"])
        ndf.ndf_field_stats(s.ctx, fid, s.mean, s.inv_norm)
        ndf.ndf_field_sorted_columns(s.ctx, fid, 0, s.mean.numel(), s.columns)
        ndf.ndf_free_ensemble(s.ctx, fid)
        return {"mean": s.mean, "inv_norm": s.inv_norm, "columns": s.columns}
    if kind == "triples":
        ndf.ndf_sample_triples(s.ctx, s.a, s.b, _measure(case), case["k"], case["n"], s.seed,
                               s.pref, s.pq, s.target)
        return {"pref": s.pref, "pq": s.pq, "target": s.target}
    if kind == "dense-step":  # the learning rate of the schedule's last stage
        loss = ndf.ndf_model_step(s.dense, s.pr, s.pq, s.target, 3e-6, True, s.grad)
        return {"loss": loss, "grad": _parts(case, s.grad)}
    if kind == "hash-step":  # the learning rate after its first decay
        loss = ndf.ndf_hash_model_step(s.hash, s.pr, s.pq, s.target, 3e-5, True, s.grad)
        return {"loss": loss, "grad": _parts(case, s.grad)}
    if kind == "dense-decode":
        ndf.ndf_infer_batch(s.dense, s.refs, s.out)
        return s.out
    ndf.ndf_hash_infer_batch(s.hash, s.refs, s.out)
    return s.out


# ---------------------------------------------------------------- exact values, in 64 bits
def _centred(f):
    """[M, N] float64 columns minus their mean, and 1 / sqrt of their sums of squares."""
    d = f.double()
    mean = d.mean(0)
    d -= mean
    ss = (d * d).sum(0)
    return d, mean, torch.where(ss > 0, ss.clamp_min(1e-300).rsqrt(), torch.zeros_like(ss))


def _ksg_pairs(x, y, k, alg):
    """KSG estimates of the pairs of rows of x and y ([P, M] float64)."""
    P, M = x.shape
    psi = torch.special.digamma(torch.arange(M + 2, device=DEVICE, dtype=torch.float64))
    out = torch.empty(P, device=DEVICE, dtype=torch.float64)
    chunk = max(1, int(2e8 / (M * M)))
    eye = torch.eye(M, dtype=torch.bool, device=DEVICE)
    for p0 in range(0, P, chunk):
        a, b = x[p0:p0 + chunk], y[p0:p0 + chunk]
        dx = (a[:, :, None] - a[:, None, :]).abs()
        dy = (b[:, :, None] - b[:, None, :]).abs()
        d = torch.maximum(dx, dy).masked_fill_(eye, math.inf)
        eps = d.topk(k, dim=2, largest=False, sorted=True).values[:, :, -1:]
        if alg == 1:
            nx = ((dx < eps) & ~eye).sum(2)
            ny = ((dy < eps) & ~eye).sum(2)
            s = (psi[nx + 1] + psi[ny + 1]).mean(1)
            out[p0:p0 + chunk] = psi[k] + psi[M] - s
        else:
            near = d <= eps
            ex = torch.where(near, dx, 0.0).amax(2, keepdim=True)
            ey = torch.where(near, dy, 0.0).amax(2, keepdim=True)
            nx = ((dx <= ex) & ~eye).sum(2)
            ny = ((dy <= ey) & ~eye).sum(2)
            out[p0:p0 + chunk] = psi[k] - 1.0 / k + psi[M] - (psi[nx] + psi[ny]).mean(1)
    return out


def _mix64(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xbf58476d1ce4e5b9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94d049bb133111eb)
    return z ^ (z >> np.uint64(31))


def _triple_positions(n, seed):
    """The documented sequence: SplitMix64 counters, 24-bit uniforms on [-1, 1)."""
    with np.errstate(over="ignore"):
        key = _mix64(np.array([int(seed)], np.uint64) ^ np.uint64(0x434f4e54504f5353))
        i = np.arange(1, 6 * n + 1, dtype=np.uint64)
        h = _mix64(key + i * np.uint64(0x9e3779b97f4a7c15)) >> np.uint64(40)
    p = torch.tensor(h.astype(np.float64) * (2.0 / 16777216.0) - 1.0, device=DEVICE).view(n, 6)
    return p[:, :3].contiguous(), p[:, 3:].contiguous()


def _corners(p, n):
    """(i0, weight) of float64 coordinates p on n corner-aligned points of [-1, 1]."""
    u = ((p + 1.0) * 0.5 * (n - 1)).clamp(0.0, n - 1.0)
    i0 = u.floor().clamp(0, max(n - 2, 0)).long()
    return i0, u - i0


def _interpolated(field, case, p):
    """[n, M] float64 columns of the field at positions p."""
    X, Y, Z = case["X"], case["Y"], case["Z"]
    flat = field.view(case["M"], -1)
    ax = [_corners(p[:, a], n) for a, n in enumerate((X, Y, Z))]
    out = torch.zeros((p.shape[0], case["M"]), dtype=torch.float64, device=DEVICE)
    for q in range(8):
        at, w = [], torch.ones(p.shape[0], dtype=torch.float64, device=DEVICE)
        for a, n in enumerate((X, Y, Z)):
            up = q >> a & 1
            at.append((ax[a][0] + up).clamp(max=n - 1))
            w = w * (ax[a][1] if up else 1.0 - ax[a][1])
        out += flat[:, (at[2] * Y + at[1]) * X + at[0]].T.double() * w[:, None]
    return out


def _dense_features(grid, case, p):
    """The corner points (row indices, weights) of every level and the features [B, 64]."""
    feats, rows, base = [], [], 0
    for res in _dense_res(case):
        ax = [_corners(p[:, a], res) for a in range(3)]
        f = 0.0
        for q in range(8):
            at, w = 0, 1.0
            for a in (2, 1, 0):
                at = at * res + ax[a][0] + (q >> a & 1)
                w = w * (ax[a][1] if q >> a & 1 else 1.0 - ax[a][1])
            rows.append((base + at, w))
            f = f + grid[base + at].double() * w[:, None]
        feats.append(f)
        base += res ** 3
    return torch.cat(feats, 1), rows


def _split_dense(params, case):
    n = sum(r ** 3 for r in _dense_res(case))
    grid = params[:n * DENSE_FEATURES].view(n, DENSE_FEATURES)
    mlp = params[n * DENSE_FEATURES:].double()
    return grid, mlp


def _dense_mlp(x, mlp):
    o = 0
    for _ in range(3):
        w = mlp[o:o + WIDTH * WIDTH].view(WIDTH, WIDTH)
        b = mlp[o + WIDTH * WIDTH:o + WIDTH * WIDTH + WIDTH]
        x = torch.relu(x @ w.T + b)
        o += WIDTH * WIDTH + WIDTH
    return x @ mlp[o:o + WIDTH] + mlp[-1]


def _output(raw, case):
    return torch.tanh(raw) if case["measure"] == "pearson" else torch.nn.functional.softplus(raw)


def _grid_positions(case, v):
    X, Y, Z = case["X"], case["Y"], case["Z"]
    v = torch.as_tensor(v, device=DEVICE)
    xyz = (v % X, v // X % Y, v // (X * Y))
    return torch.stack([-1.0 + 2.0 * i.double() / (n - 1) if n > 1 else torch.zeros_like(i, dtype=torch.float64)
                        for i, n in zip(xyz, (X, Y, Z))], 1)


def _act(x, act):
    return (x if act == 1 else 0.5 * x) + torch.sin(x) ** 2 if act else torch.relu(x)


def _hash_rows(case, p):
    """Table rows and weights of every level's corner points."""
    rows = []
    for res, entries, off, is_dense in _hash_layout(case)[0]:
        ax = [_corners(p[:, a], res) for a in range(3)]
        for q in range(8):
            i = [ax[a][0] + (q >> a & 1) for a in range(3)]
            w = 1.0
            for a in range(3):
                w = w * (ax[a][1] if q >> a & 1 else 1.0 - ax[a][1])
            if is_dense:
                at = (i[2] * res + i[1]) * res + i[0]
            else:
                at = (i[0] ^ (i[1] * 2654435761) ^ (i[2] * 805459861)) & (entries - 1)
            rows.append((off // 2 + at, w))
    return rows


def _hash_embed(p, table, rows):
    parts = [p]
    f = (2.0 ** torch.arange(12, device=DEVICE, dtype=torch.float64)) * math.pi
    for a in range(3):
        t = p[:, a:a + 1] * f
        parts.append(torch.stack([torch.sin(t), torch.cos(t)], 2).flatten(1))
    for l in range(6):
        parts.append(sum(table[at].double() * w[:, None] for at, w in rows[8 * l:8 * l + 8]))
    return torch.cat(parts, 1)


def _hash_layers(x, params, base, layers, act, last):
    for k, (w, b, c_in, c_out) in enumerate(layers):
        x = x @ params[base + w:base + b].view(c_out, c_in).T + params[base + b:base + b + c_out]
        if k < len(layers) - 1:
            x = _act(x, act)
    return x[:, 0] if last else x


def _hash_merge(a, b, mode):
    return a * b if mode == 0 else a + b if mode == 1 else (a - b).abs() if mode == 2 else torch.cat([a, b], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pearson", "pearson-batch", "ksg", "load"):
        N = case["X"] * case["Y"] * case["Z"]
        if kind == "ksg" and N * float(case["M"]) ** 2 * case["R"] > 4e9:
            return None
        fields = [f.view(case["M"], N) for f in _ensembles(case, seed)]
        a, b = fields[0], fields[-1]
        refs = _references(case, seed, case.get("R", 1))
        if kind == "ksg":
            y = b.T.double().contiguous()
            return torch.stack([_ksg_pairs(a[:, r].double().expand(N, -1), y, case["k"], case["alg"])
                                for r in refs])
        if kind == "load":
            _, mean, inv = _centred(a)
            return {"mean": mean, "inv_norm": inv, "columns": a.sort(0).values.double()}
        x, _, sx = _centred(a[:, refs])
        out = torch.empty((len(refs), N), dtype=torch.float64, device=DEVICE)
        step = max(1, int(2.5e8 / case["M"]))
        for v in range(0, N, step):
            d, _, sd = _centred(b[:, v:v + step])
            out[:, v:v + step] = (x.T @ d) * sx[:, None] * sd
        return out.clamp_(-1.0, 1.0)
    if kind == "triples":
        pr, pq = _triple_positions(case["n"], seed)
        if case["measure"] == "mi" and case["n"] * float(case["M"]) ** 2 > 4e9:
            return {"pref": pr, "pq": pq, "target": None}
        f = _ensembles(case, seed)[0]
        target = []
        for i in range(0, case["n"], 20000):
            x, y = _interpolated(f, case, pr[i:i + 20000]), _interpolated(f, case, pq[i:i + 20000])
            if case["measure"] == "mi":
                target.append(_ksg_pairs(x, y, case["k"], 1))
            else:
                (u, _, su), (v, _, sv) = _centred(x.T), _centred(y.T)
                target.append(((u * v).sum(0) * su * sv).clamp(-1.0, 1.0))
        return {"pref": pr, "pq": pq, "target": torch.cat(target)}
    if kind == "dense-decode":
        grid, mlp = _split_dense(_dense_params(case, seed), case)
        N = case["X"] * case["Y"] * case["Z"]
        fr = _dense_features(grid, case, _grid_positions(case, _references(case, seed, case["R"])))[0]
        out = torch.empty((case["R"], N), dtype=torch.float64, device=DEVICE)
        for v in range(0, N, 200000):
            fq = _dense_features(grid, case, _grid_positions(case, torch.arange(v, min(v + 200000, N))))[0]
            for r in range(case["R"]):
                out[r, v:v + 200000] = _output(_dense_mlp(torch.cat([fr[r] * fq, fr[r] + fq], 1), mlp), case)
        return out
    if kind == "dense-step":
        params = _dense_params(case, seed)
        grid, mlp = _split_dense(params, case)
        pr, pq, t = _batch(case, seed)
        fr, rr = _dense_features(grid, case, pr.double())
        fq, rq = _dense_features(grid, case, pq.double())
        with torch.enable_grad():
            fr, fq, mlp = (v.detach().requires_grad_() for v in (fr, fq, mlp))
            y = _output(_dense_mlp(torch.cat([fr * fq, fr + fq], 1), mlp), case)
            loss = (y - t.double()).abs().mean()
            loss.backward()
        g = torch.zeros(grid.shape, dtype=torch.float64, device=DEVICE)
        for f, rows in ((fr, rr), (fq, rq)):
            for i, (at, w) in enumerate(rows):
                l = i // 8 * DENSE_FEATURES
                g.index_add_(0, at, f.grad[:, l:l + DENSE_FEATURES] * w[:, None])
        return {"loss": float(loss), "grad": {"grid": g.flatten(), "mlp": mlp.grad}}
    levels, enc, dec, enc_size, n_enc, total = _hash_layout(case)
    params = _hash_params(case, seed, 0.02 if kind == "hash-step" else 0.3)
    act, merge, tables = case.get("act", 2), case.get("merge", 0), enc[0][0]
    p64 = params.double()
    side_base = (0, enc_size * (n_enc - 1))
    if kind == "hash-decode":
        N = case["X"] * case["Y"] * case["Z"]
        table = p64[:tables].view(-1, 2)

        def latent(v):
            p = _grid_positions(case, v)
            return _hash_layers(_hash_embed(p, table, _hash_rows(case, p)), p64, 0, enc, act, False)

        zr = latent(_references(case, seed, case["R"]))
        out = torch.empty((case["R"], N), dtype=torch.float64, device=DEVICE)
        for v in range(0, N, 200000):
            zq = latent(torch.arange(v, min(v + 200000, N)))
            for r in range(case["R"]):
                out[r, v:v + 200000] = _output(_hash_layers(zr[r] * zq, p64, 0, dec, act, True), case)
        return out
    pr, pq, t = _batch(case, seed)
    with torch.enable_grad():
        p64 = p64.requires_grad_()
        z, kept = [], []
        for base, pos in zip(side_base, (pr, pq)):
            rows = _hash_rows(case, pos.double())
            e = _hash_embed(pos.double(), params[base:base + tables].view(-1, 2), rows)
            e = e.detach().requires_grad_()
            kept.append((base, rows, e))
            z.append(_hash_layers(e, p64, base, enc, act, False))
        y = _output(_hash_layers(_hash_merge(z[0], z[1], merge), p64, 0, dec, act, True), case)
        loss = (y - t.double()).abs().mean()
        loss.backward()
    g = p64.grad
    for base, rows, e in kept:
        tg = g[base:base + tables].view(-1, 2)
        for i, (at, w) in enumerate(rows):
            l = 75 + i // 8 * 2
            tg.index_add_(0, at, e.grad[:, l:l + 2] * w[:, None])
    return {"loss": float(loss), "grad": _parts(case, g)}


# ---------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once, and the operations of the definitions (a k-NN
    search counted as k + 1 distances and four binary searches per member)."""
    kind = case["kind"]
    if kind in ("pearson", "pearson-batch", "ksg", "load", "triples"):
        N, M, R = case["X"] * case["Y"] * case["Z"], case["M"], case.get("R", 1)
        if kind == "load":
            return {"bytes": 8.0 * M * N + 16.0 * N, "flops": 4.0 * M * N + M * N * math.log2(M)}
        if kind == "triples":
            n, lerp = case["n"], 2 * 7 * 3.0
            per = M * (lerp + (3 * (case["k"] + 1) + 4 * math.log2(M) if case["measure"] == "mi" else 8))
            return {"bytes": 4.0 * M * min(N, 16 * n) + 28.0 * n, "flops": n * per}
        if kind == "ksg":
            return {"bytes": 4.0 * M * N + 4.0 * R * N,
                    "flops": float(R) * N * M * (3 * (case["k"] + 1) + 4 * math.log2(M))}
        return {"bytes": 4.0 * M * N + 16.0 * N + 4.0 * R * N, "flops": 2.0 * R * M * N}
    if kind == "dense-step":
        n_grid = sum(r ** 3 for r in _dense_res(case)) * DENSE_FEATURES
        mac = case["B"] * (3 * WIDTH * WIDTH + WIDTH)
        # parameters and both moments read and written, the 16-bit grid and the gradient written
        return {"bytes": 30.0 * n_grid + 28.0 * case["B"], "flops": 6.0 * mac}
    if kind == "dense-decode":
        n_grid = sum(r ** 3 for r in _dense_res(case)) * DENSE_FEATURES
        N = case["X"] * case["Y"] * case["Z"]
        return {"bytes": 2.0 * min(n_grid, 512 * N) + 4.0 * N * case["R"],
                "flops": 2.0 * N * case["R"] * (3 * WIDTH * WIDTH + WIDTH)}
    enc = 87 * WIDTH + 5 * WIDTH * WIDTH
    dec = (2 if case.get("merge", 0) == 3 else 1) * WIDTH * WIDTH + 4 * WIDTH * WIDTH + WIDTH
    total = _hash_layout(case)[5]
    if kind == "hash-step":
        return {"bytes": 28.0 * total + 28.0 * case["B"], "flops": 6.0 * case["B"] * (2 * enc + dec)}
    N = case["X"] * case["Y"] * case["Z"]
    return {"bytes": 4.0 * min(total, 96 * N) + 4.0 * N * case["R"],
            "flops": 2.0 * N * ((0 if case["mode"] == "cached" else enc) + case["R"] * dec)}
