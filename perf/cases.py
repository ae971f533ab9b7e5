"""The measured work of this library: the calls that a user of the
pass-efficient interpolative decomposition makes, through the public entry
points, from the smallest snapshot matrix to the 18.9 GB one.

Every case is a plain dict with a ``kind``:

  id        stream the snapshots, randomized ID, sub-sampled ID, error pass
  sketch    stream the snapshots of one run: W = Psi A, Y = A Omega, A_c
  error     reconstruction error of a finished ID over the whole matrix
  single    single-pass ID: lifted skeleton and its error
  batch     many uneven matrices in one launch
  train     one training step of the learned proposal's network
  propose   learned proposal and the pivoted QR restricted to it

Inputs are turbulence-like fields: 64 Fourier modes in x and z with wall
profiles in y, amplitudes |kappa|^(-5/3), every mode convected at its own speed
with a slow envelope, unit RMS, plus 1e-6 noise.
"""
import math
import random

import numpy as np
import torch

from paper_1905_13257_gb300 import IdBatch, IdSketch, Mlp
from paper_1905_13257_gb300.learned import LearnedProposal

DEV = "cuda"


# ------------------------------------------------------------------- cases

def listed():
    """The listed cases, smallest first within each part of the library."""
    return [
        # a first try on a toy grid, every chunk processed as it arrives:
        # latency, launches and host work decide
        dict(name="id_small", kind="id", nx=16, ny=12, nz=16, ncomp=3, n=96, k=8, l=16, stride=2,
             dtype="f32", window=0),
        # an odd grid straight from a solver: no column but the first is
        # aligned, ragged tiles everywhere
        dict(name="id_odd", kind="id", nx=65, ny=49, nz=33, ncomp=3, n=333, k=50, l=60, stride=2,
             dtype="f32", window=333),
        # double-precision snapshots of a 32^3 box (the FP64 configuration of
        # the test suite)
        dict(name="id_f64", kind="id", nx=32, ny=32, nz=32, ncomp=3, n=200, k=20, l=30, stride=4,
             dtype="f64", window=0),
        # the ordinary whole call: 1000 snapshots of a 64 x 48 x 64 channel,
        # sub-sampled by 2
        dict(name="id_channel", kind="id", nx=64, ny=48, nz=64, ncomp=3, n=1000, k=50, l=60,
             stride=2, dtype="f32", window=1000),
        # the benchmark's matrix: both sketches and the coarse rows of 18.9 GB
        dict(name="sketch_large", kind="sketch", nx=128, ny=96, nz=128, ncomp=3, n=1000, k=50,
             l=60, stride=4, prec="exact", want_Y=True, buffers="one"),
        # in-situ use: the solver hands over each chunk of 32 snapshots in a
        # buffer of its own
        dict(name="sketch_chunks", kind="sketch", nx=64, ny=48, nz=64, ncomp=3, n=512, k=50, l=60,
             stride=4, prec="exact", want_Y=True, buffers="own"),
        # the FP8 precision form, W only
        dict(name="sketch_fp8", kind="sketch", nx=96, ny=65, nz=96, ncomp=3, n=500, k=50, l=60,
             stride=0, prec="fp8", want_Y=False, buffers="one"),
        # checking a finished compression against all of the benchmark's data
        dict(name="error_large", kind="error", nx=128, ny=96, nz=128, ncomp=3, n=1000, k=50,
             dtype="f32"),
        # Algorithm 6 on a grid whose y direction ends past its last coarse plane
        dict(name="single_pass", kind="single", nx=96, ny=66, nz=96, ncomp=3, n=256, k=40,
             stride=4),
        # block-wise compression: 12 matrices of the batched benchmark's mix
        dict(name="batch_mixed", kind="batch", count=12, ny_min=17, ny_max=36, n_min=64, n_max=512,
             k_max=80, mix=1),
        # the learned proposal: training step, and scoring plus restricted QR
        dict(name="train_step", kind="train", n=512, features=4096, hidden=256),
        dict(name="propose", kind="propose", grid=32, n=512, k=50, l=60, hidden=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["id", "id", "id", "sketch", "sketch", "error", "single", "batch", "train",
                       "propose"])
    if kind == "id":
        f64 = rng.random() < 0.3
        top = 34 if f64 else 72
        nx, ny, nz = (rng.randint(12, top) for _ in range(3))
        if rng.random() < 0.6:
            nx = 4 * max(3, nx // 4)
        n = _log_int(rng, 48, 250 if f64 else 1000)
        k = rng.randint(6, min(50, n // 3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, ncomp=3, n=n, k=k, l=k + 10,
                    stride=rng.choice([2, 4]), dtype="f64" if f64 else "f32",
                    window=rng.choice([0, n]))
    if kind == "sketch":
        nx = 4 * rng.randint(10, 32)
        n = _log_int(rng, 40, 1000)
        prec = rng.choice(["exact", "exact", "bf16", "fp8"])
        want_Y = rng.random() < 0.6
        k = rng.randint(10, min(50, n // 3))
        return dict(kind=kind, nx=nx, ny=rng.randint(30, 90), nz=rng.randint(40, 120), ncomp=3,
                    n=n, k=k, l=k + 10, stride=rng.choice([0, 2, 4]), prec=prec, want_Y=want_Y,
                    buffers=rng.choice(["one", "own"]))
    if kind == "error":
        f64 = rng.random() < 0.25
        n = _log_int(rng, 60, 250 if f64 else 1000)
        return dict(kind=kind, nx=rng.randint(16, 32 if f64 else 120), ny=rng.randint(16, 40),
                    nz=rng.randint(16, 32 if f64 else 120), ncomp=3, n=n,
                    k=rng.randint(5, min(64, n // 2)), dtype="f64" if f64 else "f32")
    if kind == "single":
        n = _log_int(rng, 60, 400)
        return dict(kind=kind, nx=4 * rng.randint(6, 26), ny=rng.randint(20, 70),
                    nz=rng.randint(24, 100), ncomp=3, n=n, k=rng.randint(8, min(60, n // 3)),
                    stride=rng.choice([2, 3, 4]))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 14), ny_min=12, ny_max=rng.randint(16, 38),
                    n_min=64, n_max=rng.randint(100, 512), k_max=rng.randint(20, 80),
                    mix=rng.randint(2, 10 ** 6))
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 100, 1000), features=_log_int(rng, 500, 6000),
                    hidden=rng.choice([96, 128, 200, 256]))
    n = rng.randint(256, 700)
    k = rng.randint(16, 50)
    return dict(kind=kind, grid=2 * rng.randint(10, 18), n=n, k=k, l=k + 10,
                hidden=rng.choice([128, 256]))


# ------------------------------------------------------------------ inputs

LX, LZ = 4.0 * math.pi, 4.0 * math.pi / 3.0


def _generator(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _wall_normal(ny):
    if ny == 1:
        return np.zeros(1)
    return np.tanh(2.0 * (2.0 * np.arange(ny) / (ny - 1) - 1.0)) / math.tanh(2.0)


def _grid_of(case):
    if "grid" in case:
        return (case["grid"],) * 3 + (3,)
    return case["nx"], case["ny"], case["nz"], case["ncomp"]


def _field(nx, ny, nz, ncomp, n, seed, dtype=torch.float32):
    """Snapshot matrix (m x n, column-major view), row r = ((c ny + j) nz + k) nx + i."""
    g = torch.Generator()
    g.manual_seed(int(seed) * 7919 + 11)
    work = torch.float64 if dtype == torch.float64 else torch.float32
    kx, kz = [t.reshape(-1).double() for t in
              torch.meshgrid(torch.arange(1, 9), torch.arange(1, 9), indexing="ij")]
    ax, az = 2 * math.pi * kx / LX, 2 * math.pi * kz / LZ
    amp = torch.hypot(ax, az) ** (-5.0 / 3.0)
    q = ((kx + kz) % 4)
    phase = 2 * math.pi * torch.rand(64, ncomp, generator=g, dtype=torch.float64)
    speed = 0.8 * (0.75 + 0.5 * torch.rand(64, generator=g, dtype=torch.float64))
    shift = torch.rand(64, generator=g, dtype=torch.float64)
    t = torch.arange(n, dtype=torch.float64) * (8.0 * LX / (0.8 * n))
    env = 1.0 + 0.5 * torch.sin(2 * math.pi * (shift[:, None] + t[None] / (8.0 * LX / 0.8)))
    om = (ax * speed)[:, None] * t[None]
    T = torch.cat([env * torch.cos(om), env * torch.sin(om)]).to(DEV, work)      # 128 x n
    y = torch.from_numpy(_wall_normal(ny))
    cheb = torch.cos(q[:, None] * torch.arccos(y.clamp(-1, 1))[None])
    th = (az[:, None] * (torch.arange(nz) * (LZ / nz)))[:, :, None] + \
        (ax[:, None] * (torch.arange(nx) * (LX / nx)))[:, None, :]
    plane = ny * nz * nx
    At = torch.empty((n, ncomp * plane), dtype=dtype, device=DEV)
    norm = 0.0
    for c in range(ncomp):
        prof = (amp[:, None] * (1 - y * y)[None] ** (2 if c == 1 else 1) * cheb).to(DEV, work)
        ang = (th + phase[:, c, None, None]).to(DEV, work).reshape(64, -1)
        S = torch.cat([(prof[:, :, None] * f(ang)[:, None, :]).reshape(64, -1)
                       for f in (torch.cos, torch.sin)])                         # 128 x plane
        norm = norm + ((S @ S.T).double() * (T @ T.T).double()).sum()
        torch.matmul(T.T, S, out=At[:, c * plane:(c + 1) * plane])
        del S
    scale = 1.0 / torch.sqrt(norm / (ncomp * plane * n))
    gen = _generator(seed)
    step = max(1, (1 << 28) // (ncomp * plane))
    for j in range(0, n, step):
        blk = At[j:j + step]
        blk.mul_(scale.to(dtype)).add_(torch.randn(blk.shape, dtype=dtype, device=DEV,
                                                   generator=gen), alpha=1e-6)
    return At.T


def _dtype(case):
    return torch.float64 if case.get("dtype") == "f64" else torch.float32


def _matrix(case, seed):
    return _field(*_grid_of(case), case["n"], seed, _dtype(case))


def _batch_problems(case, seed):
    """The batch's matrices: m = 12 ny^3 rows, every other one in the BF16 form."""
    r = random.Random(case["mix"])
    out = []
    for b in range(case["count"]):
        ny = r.randint(case["ny_min"], case["ny_max"])
        n = r.randint(case["n_min"], case["n_max"])
        k = r.randint(10, min(case["k_max"], n - 10))
        A = None
        if seed is not None:
            A = _field(2 * ny, ny, 2 * ny, 3, n, seed * 131 + b)
        out.append(dict(A=A, m=12 * ny ** 3, n=n, k=k, l=min(k + 10, n), seed=b + 1,
                        prec="bf16" if b % 2 else "exact"))
    return out


def _finished_id(A, k):
    """k spread-out columns and the least-squares P over a row sample, as an
    earlier run of the decomposition leaves them."""
    m, n = A.shape
    J = torch.linspace(0, n - 1, k, device=DEV).round().long()
    rows = torch.linspace(0, m - 1, min(m, 4096), device=DEV).long()
    s = A[rows].double()
    P = torch.linalg.lstsq(s[:, J], s).solution
    P[:, J] = torch.eye(k, dtype=torch.float64, device=DEV)
    return J, P


def _network(case, seed, F):
    g = _generator(seed, 5)
    H = case["hidden"]
    return {"W1": torch.randn(F, H, device=DEV, generator=g) / math.sqrt(F),
            "b1": 0.1 * torch.randn(H, device=DEV, generator=g),
            "w2": torch.randn(H, device=DEV, generator=g) / math.sqrt(H),
            "b2": 0.1 * torch.randn(1, device=DEV, generator=g)}


def _train_data(case, seed):
    """Feature rows of consecutive snapshots and the skeleton's labels."""
    g = _generator(seed, 6)
    n, F = case["n"], case["features"]
    t = torch.linspace(0, 6.0, n, device=DEV)[:, None] * \
        (0.5 + torch.rand(1, 24, device=DEV, generator=g)) + \
        6.0 * torch.rand(1, 24, device=DEV, generator=g)
    X = torch.cos(t) @ torch.randn(24, F, device=DEV, generator=g) / math.sqrt(12.0)
    y = (torch.rand(n, device=DEV, generator=g) < 0.1).float()
    return X, y


def _mesh(case):
    nx, ny, nz, _ = _grid_of(case)
    return (np.arange(nx) * (LX / nx), _wall_normal(ny), np.arange(nz) * (LZ / nz)), (LX, 0.0, LZ)


def _handle(case, seed, m, dtype=torch.float32, **kw):
    if case.get("stride"):
        nx, ny, nz, nc = _grid_of(case)
        kw.update(grid=(nx, ny, nz), ncomp=nc, coarse_stride=(case["stride"],) * 3,
                  want_coarse=True)
    return IdSketch(m, case["n"], case["k"], case["l"], seed=seed, dtype=dtype, **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "id":
        A = _matrix(case, seed)
        sk = _handle(case, seed, A.shape[0], A.dtype, want_Y=True, window_cols=case["window"])
        return dict(kind=kind, A=A, sk=sk)
    if kind == "sketch":
        A = _matrix(case, seed)
        chunks = [A[:, j:j + 32] for j in range(0, case["n"], 32)]
        if case["buffers"] == "own":
            chunks = [c.T.clone().T for c in chunks]
            A = None
        m = chunks[0].shape[0]
        sk = _handle(case, seed, m, want_Y=case["want_Y"], prec=case["prec"],
                     window_cols=case["n"])
        return dict(kind=kind, chunks=chunks, sk=sk)
    if kind == "error":
        A = _matrix(case, seed)
        J, P = _finished_id(A, case["k"])
        sk = IdSketch(A.shape[0], case["n"], case["k"], case["k"], dtype=A.dtype, want_Y=False)
        return dict(kind=kind, A=A, sk=sk, J=J.int(), P=P)
    if kind == "single":
        A = _matrix(case, seed)
        sk = _handle(dict(case, l=case["k"]), seed, A.shape[0], want_Y=False)
        sk.stream_columns(A)
        Jc, Pc, kc = sk.coarse_factor()
        xyz, per = _mesh(case)
        sk.set_mesh(*xyz, per)
        return dict(kind=kind, A=A, sk=sk, Jc=Jc, Pc=Pc)
    if kind == "batch":
        return dict(kind=kind, bt=IdBatch(_batch_problems(case, seed)))
    if kind == "train":
        X, y = _train_data(case, seed)
        return dict(kind=kind, X=X, y=y, net=Mlp(_network(case, seed, case["features"])))
    if kind == "propose":
        A = _matrix(case, seed)
        g = case["grid"]
        st = max(1, g // 16)
        prop = LearnedProposal((g, g, g), case["k"], hidden=case["hidden"], stride=(st, st, st))
        prop.net = Mlp(_network(case, seed, prop.F))
        prop.features(A)        # sets the feature scale, as the first window does
        sk = _handle(case, seed, A.shape[0], want_Y=False)
        sk.stream_columns(A)
        return dict(kind=kind, A=A, sk=sk, prop=prop)
    raise ValueError(kind)


# -------------------------------------------------------------------- runs

def _sketches(sk):
    """The handle's own buffers W, Y and A_c; each keeps its handle alive."""
    out = sk.sketches()
    for t in out:
        if t is not None:
            t.handle = sk
    return out


def run(state):
    kind, sk = state["kind"], state.get("sk")
    if kind == "id":
        A = state["A"]
        sk.reset()
        for j in range(0, A.shape[1], 32):
            sk.stream_columns(A[:, j:j + 32])
        J, P, _ = sk.factor()
        Jc, Pc, _ = sk.coarse_factor()
        fro, mx = sk.reconstruct_error(A, J, P)
        W, Y, Ac = _sketches(sk)
        return dict(J=J, P=P, Jc=Jc, Pc=Pc, fro=fro, mx=mx, W=W, Y=Y, Ac=Ac)
    if kind == "sketch":
        sk.reset()
        for c in state["chunks"]:
            sk.stream_columns(c)
        sk.flush()
        W, Y, Ac = _sketches(sk)
        return dict(W=W, Y=Y, Ac=Ac)
    if kind == "error":
        fro, mx = sk.reconstruct_error(state["A"], state["J"], state["P"])
        return dict(fro=fro, mx=mx)
    if kind == "single":
        S = sk.single_pass_lift(state["Jc"])
        fro, mx = sk.single_pass_error(state["A"], state["Jc"], state["Pc"])
        return dict(S=S, fro=fro, mx=mx)
    if kind == "batch":
        state["bt"].run()
        return [dict(J=J, P=P) for J, P, _ in state["bt"].wait()]
    if kind == "train":
        net = state["net"]
        s = net.forward(state["X"])
        g = net.backward(state["X"], state["y"], 9.0)
        net.step(g, 0.05)
        return dict(s=s, grads=g, W1=net.W1, b1=net.b1, w2=net.w2, b2=net.b2)
    X = state["prop"].features(state["A"])
    cand = state["prop"].propose(X)
    J, P, _ = sk.factor_restricted(cand)
    return dict(X=X, s=state["prop"].net.s, cand=cand, J=J, P=P)


# -------------------------------------------------------------------- work

def work(case):
    """Bytes: inputs read once and outputs written once.  Flops: the products
    of the sketches, the k steps of each pivoted QR (two products with the
    matrix per step), the reconstruction."""
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for p in _batch_problems(case, None):
            b += 4.0 * p["m"] * p["n"] + 8.0 * p["k"] * p["n"]
            f += 2.0 * p["m"] * p["n"] * p["l"] + 4.0 * p["l"] * p["n"] * p["k"]
        return dict(bytes=b, flops=f)
    if kind == "train":
        n, F, H = case["n"], case["features"], case["hidden"]
        return dict(bytes=4.0 * (n * F + 3 * F * H + 2 * n), flops=4.0 * n * F * H + 20.0 * n * H)
    nx, ny, nz, nc = _grid_of(case)
    m, n, k = nx * ny * nz * nc, case["n"], case["k"]
    e = 8 if case.get("dtype") == "f64" else 4
    l, s = case.get("l", k), case.get("stride", 0)
    mc = nc * -(-nx // s) * -(-ny // s) * -(-nz // s) if s else 0
    if kind == "id":
        # read by the sketch and again by the error pass, which needs its result
        return dict(bytes=2.0 * e * m * n + e * m * l + e * mc * n + 16.0 * k * n + 8.0 * l * n,
                    flops=4.0 * m * n * l + 2.0 * m * n * k + 4.0 * (mc + l) * n * k)
    if kind == "sketch":
        y = 1 if case["want_Y"] else 0
        return dict(bytes=4.0 * (m * n + y * m * l + mc * n) + 8.0 * l * n,
                    flops=2.0 * (1 + y) * m * n * l)
    if kind == "error":
        return dict(bytes=float(e) * m * n + 8.0 * k * n, flops=2.0 * m * n * k)
    if kind == "single":
        return dict(bytes=4.0 * (m * n + m * k + mc * k) + 8.0 * k * n,
                    flops=2.0 * m * n * k + 16.0 * m * k)
    F, H = len(range(0, nx, max(1, nx // 16))) ** 3, case["hidden"]
    return dict(bytes=4.0 * (2 * n * F + F * H) + 8.0 * (l + k) * n,
                flops=2.0 * n * F * H + 4.0 * l * n * k)


# ------------------------------------------------- the same in 64 bits

def _philox(c, key):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    m32 = 0xFFFFFFFF
    c0, c1, c2, c3 = c
    k0, k1 = key & m32, (key >> 32) & m32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & m32) ^ c1 ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c3 ^ k1,
                          p0 & m32)
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c0, c1, c2, c3


def _gauss(index, width, stream, seed):
    """G(i, s) of include/idsketch.h for the indices given: len x width, FP64."""
    u = (torch.arange(4096, dtype=torch.float64, device=DEV) + 0.5) / 4096
    table = torch.special.ndtri(u).to(torch.bfloat16).double()
    cols = []
    for sb in range(-(-width // 10)):
        x = _philox((index & 0xFFFFFFFF, index >> 32, torch.full_like(index, sb),
                     torch.full_like(index, stream)), seed) + (torch.zeros_like(index),)
        for f in range(10):
            w, o = divmod(12 * f, 32)
            cols.append(table[((x[w] >> o) | (x[w + 1] << (32 - o))) & 0xFFF])
    return torch.stack(cols[:width], 1)


def _exact_sketches(A, l, seed, want_Y=True, rounded=lambda x, r: x.double()):
    m, n = A.shape
    W = torch.zeros(l, n, dtype=torch.float64, device=DEV)
    om = _gauss(torch.arange(n, device=DEV), l, 2, seed)
    Y = torch.empty(l, m, dtype=torch.float64, device=DEV).T if want_Y else None
    step = max(1024, (1 << 26) // n)
    for r in range(0, m, step):
        a = rounded(A[r:r + step], r)
        W += _gauss(torch.arange(r, r + a.shape[0], device=DEV), l, 1, seed).T @ a
        if want_Y:
            Y[r:r + step] = a @ om
    return W, Y


def _exact_id(B, k, cand=None):
    """k-step column-pivoted Householder QR of B (over the columns cand) -> J, P."""
    B = B.double().clone()
    n = B.shape[1]
    J = []
    free = torch.zeros(n, dtype=torch.bool, device=DEV)
    free[slice(None) if cand is None else cand.long()] = True
    for s in range(k):
        p = int(torch.where(free, B[s:].square().sum(0), -1.0).argmax())
        J.append(p)
        free[p] = False
        v = B[s:, p].clone()
        beta = -torch.copysign(v.norm(), v[0])
        v[0] -= beta
        B[s:] -= torch.outer(v * (2.0 / v.square().sum()), v @ B[s:])
    J = torch.tensor(J, device=DEV)
    P = torch.linalg.solve_triangular(B[:k, J].triu(), B[:k], upper=True)
    P[:, J] = torch.eye(k, dtype=torch.float64, device=DEV)
    return J.int(), P


def _exact_error(A, skeleton, P):
    m, n = A.shape
    res = tot = 0.0
    mx = 0.0
    step = max(1024, (1 << 26) // n)
    for r in range(0, m, step):
        a = A[r:r + step].double()
        e = a - skeleton(r, r + a.shape[0]) @ P
        res, tot = res + e.square().sum(), tot + a.square().sum()
        mx = max(mx, float(torch.where(a != 0, e.abs() / a.abs(), 0.0).max()))
    return float(torch.sqrt(res / tot)), mx


def _coarse_rows(case):
    nx, ny, nz, nc = _grid_of(case)
    s = case["stride"]
    ax = [torch.arange(0, d, s, device=DEV) for d in (ny, nz, nx)]
    c = torch.arange(nc, device=DEV)
    return (((c[:, None, None, None] * ny + ax[0][:, None, None]) * nz + ax[1][:, None]) * nx +
            ax[2]).reshape(-1)


def _interp(x, stride, period):
    """Coarse neighbours and weight of every index of one direction."""
    n = len(x)
    c = -(-n // stride)
    lo, hi, w = np.zeros(n, int), np.zeros(n, int), np.zeros(n)
    for i in range(n):
        a = i // stride
        lo[i] = hi[i] = a
        if i % stride:
            if a + 1 < c:
                hi[i], x1 = a + 1, x[(a + 1) * stride]
            elif period > 0:
                hi[i], x1 = 0, x[0] + period
            elif c > 1:
                lo[i], hi[i], x1 = c - 2, c - 1, x[(c - 1) * stride]
            else:
                continue
            w[i] = (x[i] - x[lo[i] * stride]) / (x1 - x[lo[i] * stride])
    return [torch.as_tensor(v, device=DEV) for v in (lo, hi, w)]


def _exact_lift(case, Sc):
    """M A_c(:, J_c): trilinear interpolation along x, z and y, m x k."""
    nx, ny, nz, nc = _grid_of(case)
    s, k = case["stride"], Sc.shape[1]
    f = Sc.reshape(nc, -(-ny // s), -(-nz // s), -(-nx // s), k)
    (x, y, z), per = _mesh(case)
    for dim, coord, p in ((3, x, per[0]), (2, z, per[2]), (1, y, per[1])):
        lo, hi, w = _interp(coord, s, p)
        w = w.reshape([-1 if d == dim else 1 for d in range(5)])
        f = f.index_select(dim, lo) * (1 - w) + f.index_select(dim, hi) * w
    return f.reshape(-1, k)


def _e4m3(A):
    """Entries of A rounded to E4M3 under each column's power-of-two scale."""
    mx = A.abs().amax(0).double()
    e = torch.floor(torch.log2(448.0 / mx.clamp_min(1e-300)))
    e = torch.where(mx * torch.exp2(e) > 448.0, e - 1, e)
    e = torch.where(mx * torch.exp2(e + 1) <= 448.0, e + 1, e).clamp(-100, 100)
    sc = torch.exp2(torch.where(mx > 0, e, 0.0))
    return lambda a, r: (a.double() * sc).float().to(torch.float8_e4m3fn).double() / sc


def _bf16(x):
    return x.to(torch.bfloat16).double()


def _gelu_net(X, p):
    z = _bf16(X) @ _bf16(p["W1"]) + p["b1"].double()
    cdf = 0.5 * (1.0 + torch.erf(z / math.sqrt(2.0)))
    return z, cdf, z * cdf, (z * cdf) @ p["w2"].double() + p["b2"].double()


def exact(case, seed):
    """What run() returns, in 64 bits (the precision forms: of the rounded data)."""
    kind = case["kind"]
    if kind == "id":
        A = _matrix(case, seed)
        W, Y = _exact_sketches(A, case["l"], seed)
        J, P = _exact_id(W, case["k"])
        Ac = A[_coarse_rows(case)]
        Jc, Pc = _exact_id(Ac, case["k"])
        fro, mx = _exact_error(A, lambda r, q: A[r:q, J.long()].double(), P)
        return dict(J=None, P=P, Jc=None, Pc=Pc, fro=fro, mx=mx, W=W, Y=Y,
                    Ac=Ac.double().T.contiguous().T)
    if kind == "sketch":
        A = _matrix(case, seed)
        rounded = {"exact": lambda x, r: x.double(), "bf16": lambda x, r: _bf16(x),
                   "fp8": _e4m3(A) if case["prec"] == "fp8" else None}[case["prec"]]
        W, Y = _exact_sketches(A, case["l"], seed, case["want_Y"], rounded)
        Ac = A[_coarse_rows(case)].double() if case.get("stride") else None
        return dict(W=W, Y=Y, Ac=Ac)
    if kind == "error":
        A = _matrix(case, seed)
        J, P = _finished_id(A, case["k"])
        fro, mx = _exact_error(A, lambda r, q: A[r:q, J].double(), P)
        return dict(fro=fro, mx=mx)
    if kind == "single":
        A = _matrix(case, seed)
        Ac = A[_coarse_rows(case)]
        Jc, Pc = _exact_id(Ac, case["k"])
        S = _exact_lift(case, Ac[:, Jc.long()].double())
        fro, mx = _exact_error(A, lambda r, q: S[r:q], Pc)
        return dict(S=S, fro=fro, mx=mx)
    if kind == "batch":
        out = []
        for p in _batch_problems(case, seed):
            rounded = (lambda x, r: _bf16(x)) if p["prec"] == "bf16" else (lambda x, r: x.double())
            W, _ = _exact_sketches(p["A"], p["l"], p["seed"], False, rounded)
            out.append(dict(J=None, P=_exact_id(W, p["k"])[1]))
            p["A"] = None
        return out
    if kind == "train":
        X, y = _train_data(case, seed)
        p = _network(case, seed, case["features"])
        z, cdf, G, s = _gelu_net(X, p)
        sg, n = torch.sigmoid(s), X.shape[0]
        ds = (-9.0 * y * (1.0 - sg) + (1.0 - y) * sg) / n
        dz = ds[:, None] * p["w2"].double() * \
            (cdf + z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi))
        g = {"W1": _bf16(X).T @ _bf16(dz.float()), "b1": dz.sum(0), "w2": G.T @ ds,
             "b2": ds.sum().reshape(1)}
        new = {k: p[k].double() - 0.05 * g[k] for k in g}
        return dict(s=s, grads=g, **new)
    A = _matrix(case, seed)
    gr, st = case["grid"], max(1, case["grid"] // 16)
    i = torch.arange(0, gr, st, device=DEV)
    rows = ((i[:, None, None] * gr + i[:, None]) * gr + i).reshape(-1)
    X = A[rows].T
    X = X * torch.tensor(1.0 / math.sqrt(float(X.double().square().mean())), dtype=torch.float32,
                         device=DEV)
    s = _gelu_net(X, _network(case, seed, rows.numel()))[3]
    n, k = case["n"], case["k"]
    cand = torch.cat([q * n // k + s[q * n // k:(q + 1) * n // k].topk(2).indices.sort().values
                      for q in range(k)])
    W, _ = _exact_sketches(A, case["l"], seed, False)
    J, P = _exact_id(W, k, cand)
    return dict(X=X.double(), s=s, cand=None, J=None, P=P)
