"""Cases that stand for the work of this library in use: per-frequency solves,
their single operator applications and gradients, the dense adjoint, the data
step of a new frequency, the warm-start stage and the time <-> frequency
transforms, each through the public binding.

Inputs are seeded: D has a spectrum decaying from 1 to 1e-3, U = D X + noise at
a stated SNR with X a planted tile low-rank matrix whose energy sits near the
diagonal, start points are small random factors.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2412_14973_gb300 as T

_PREC = {"fp32": T.TLR_PREC_FP32, "bf16x3": T.TLR_PREC_BF16X3, "tf32": T.TLR_PREC_TF32}
_DIAG = {"rule": T.TLR_DIAG_RULE, "lowrank": T.TLR_DIAG_LOWRANK, "dense": T.TLR_DIAG_DENSE}
_DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(name, kind, nx, ny, ns, tile, rank, prec, **more):
    c = dict(kind=kind, nx=nx, ny=ny, ns=ns, tile=tile, tile2=0, rank=rank, prec=prec, diag="rule", general=False,
             snr=10.0, stages=3)
    c.update(more)
    return dict(c, name=name) if name else c


def _stack(name, ntr, nt, f0, nf):
    c = dict(kind="stack", ntr=ntr, nt=nt, f0=f0, nf=nf)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one frequency of a small survey, solved again and again by an interactive program: launch latency
        _case("solve_nr256", "solve", 16, 16, 256, 64, 8, "bf16x3", diag="dense", snr=20.0),
        # a sparse survey (30 % of the sources dropped) in the library's default precision
        _case("solve_nr1024_fp32", "solve", 32, 32, 717, 128, 12, "fp32", diag="lowrank", snr=5.0),
        # a frequency of the batched survey: the first lambda stage (10 of the 30 iterations)
        _case("solve_nr4096", "solve", 64, 64, 4096, 256, 26, "bf16x3", stages=1),
        # misfit and gradient of the largest survey (mean rank), as an outer optimiser calls them
        _case("grad_nr9216", "grad", 96, 96, 9216, 384, 36, "bf16x3"),
        # the same in the default precision at the batched survey's size
        _case("grad_nr4096_fp32", "grad", 64, 64, 4096, 256, 26, "fp32"),
        # the general (non-reciprocal) form on unequal tiles
        _case("grad_general_tiles", "grad", 64, 32, 1843, 192, 26, "bf16x3", tile2=320, general=True),
        # forward modelling, TF32, odd receiver grid and source count
        _case("apply_odd_tf32", "apply", 45, 45, 1501, 135, 17, "tf32", diag="lowrank"),
        # the dense adjoint G = V D^H (imaging condition)
        _case("adjoint_nr4096", "adjoint", 64, 64, 4096, 256, 26, "bf16x3"),
        # the data step of one more frequency: handle from raw D, U, its panels read back, handle destroyed
        _case("create_nr2048", "create", 64, 32, 2048, 128, 16, "bf16x3"),
        # warm-start stage, first half: the benchmark solution, 20 conjugate-gradient steps
        _case("benchmark_nr2048", "benchmark", 64, 32, 2048, 256, 16, "bf16x3"),
        # warm-start stage, second half: tile ranks of a benchmark solution, then the SVD / Takagi start factors
        _case("warm_nr1536", "warm", 48, 32, 768, 128, 16, "fp32", diag="lowrank"),
        # field records to a frequency band and back: 4.5 s at 4 ms
        _stack("stack_nt1125", 40000, 1125, 10, 200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    # no dearer than the largest listed solve; the CUDA-core products of the default precision are about 12 times slower
    most = next(work(c)["flops"] for c in listed() if c["name"] == "solve_nr4096")
    while True:
        c = _drawn(rng)
        if work(c)["flops"] * (12 if c.get("prec") == "fp32" and c["kind"] != "warm" else 1) <= most:
            return c


def _drawn(rng):
    kind = rng.choice(["solve", "solve", "grad", "grad", "grad", "apply", "apply", "adjoint", "create", "benchmark",
                       "warm", "stack"])
    if kind == "stack":
        nt = _log(rng, 64, 2048)
        f0 = rng.randrange(0, nt // 8)
        nf = rng.randrange(1, nt // 2 + 2 - f0)
        return _stack(None, _log(rng, 500, min(100000, 40000 * 1125 // nt)), nt, f0, nf)
    # a receiver grid of Nx x Ny tiles of tx x ty receivers
    most = {"solve": 4096, "grad": 9216, "apply": 9216, "adjoint": 4096, "create": 4096, "benchmark": 2048,
            "warm": 1536}[kind]
    while True:
        tx, ty, mx, my = rng.randrange(6, 21), rng.randrange(6, 21), rng.randrange(2, 6), rng.randrange(2, 6)
        nr = tx * ty * mx * my
        if 256 <= nr <= most and (kind != "warm" or tx * ty <= 160):
            break
    tile, tile2 = tx * ty, 0
    prec = rng.choice(["bf16x3", "bf16x3", "fp32"] if kind in ("solve", "benchmark") else
                      ["bf16x3", "bf16x3", "fp32", "tf32"])
    general = kind in ("grad", "apply") and rng.random() < 0.25
    if kind in ("grad", "apply") and mx * my % 2 == 0 and rng.random() < 0.3:
        tile2 = tile + rng.randrange(1, tile // 2)      # pairs of unequal tiles of the same sum
        tile = 2 * tile - tile2
    rank = min(_log(rng, 2, 64), min(tile, tile2 or tile) // 2)
    ns = max(64, min(int(nr * rng.uniform(0.5, 1.2)), 9216))
    diag = rng.choice(["rule", "lowrank", "dense"])
    return _case(None, kind, tx * mx, ty * my, ns, tile, rank, prec, tile2=tile2, diag=diag, general=general,
                 snr=rng.choice([5.0, 10.0, 20.0]), stages=1 if nr > 700 else 3)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _tiles(c):
    nr = c["nx"] * c["ny"]
    if not c["tile2"]:
        return [c["tile"]] * (nr // c["tile"])
    return [c["tile"], c["tile2"]] * (nr // (c["tile"] + c["tile2"]))


def _dense(c):
    return [c["diag"] == "dense" or (c["diag"] == "rule" and 4 * c["rank"] >= d) for d in _tiles(c)]


def _pairs(c):
    n = len(_tiles(c))
    return [(i, j) for j in range(n) for i in range(n) if (i != j if c["general"] else i > j)]


def _blocks(c):
    """(kind, i, j, rows, columns) of every block of theta in stacking order."""
    d, dense, k = _tiles(c), _dense(c), c["rank"]
    out = []
    for i, di in enumerate(d):
        if dense[i]:
            out.append(("Z", i, i, di, di))
        elif c["general"]:
            out += [("QL", i, i, di, k), ("QR", i, i, di, k)]
        else:
            out.append(("Q", i, i, di, k))
    out += [("L", i, j, d[i], k) for i, j in _pairs(c)]
    out += [("R", i, j, d[j], k) for i, j in _pairs(c)]
    return out


def _factors(c, theta):
    """The blocks of theta as matrices: {(kind, i, j): block}."""
    o, out = 0, {}
    for kind, i, j, r, k in _blocks(c):
        out[kind, i, j] = theta[o:o + r * k].view(r, k)
        o += r * k
    return out


def _randn(g, *shape):
    return torch.randn(*shape, dtype=torch.complex64, device=_DEV, generator=g)


def _theta(c, g):
    """Factors of a planted X: CN(0, 1) / sqrt(d k), falling off from the diagonal."""
    parts = []
    for kind, i, j, r, k in _blocks(c):
        a = _randn(g, r, k) / math.sqrt(r * (1 if kind == "Z" else k)) / (1 + abs(i - j))
        parts.append((0.5 * (a + a.T) if kind == "Z" else a).reshape(-1))
    return torch.cat(parts)


def _rows(c):
    at = np.concatenate([[0], np.cumsum(_tiles(c))])
    return [slice(int(a), int(b)) for a, b in zip(at[:-1], at[1:])]


def _assemble(c, theta):
    """X_h from its factors."""
    nr, rows, f = c["nx"] * c["ny"], _rows(c), _factors(c, theta)
    X = torch.empty((nr, nr), dtype=theta.dtype, device=theta.device)
    for i, ri in enumerate(rows):
        if ("Z", i, i) in f:
            Z = f["Z", i, i]
            X[ri, ri] = Z if c["general"] else 0.5 * (Z + Z.T)
        elif c["general"]:
            X[ri, ri] = f["QL", i, i] @ f["QR", i, i].T
        else:
            X[ri, ri] = f["Q", i, i] @ f["Q", i, i].T
    for i, j in _pairs(c):
        X[rows[i], rows[j]] = f["L", i, j] @ f["R", i, j].T
        if not c["general"]:
            X[rows[j], rows[i]] = X[rows[i], rows[j]].T
    return X


def _hilbert(nx, ny):
    """Natural indices (y nx + x) of the grid's receivers along the Hilbert curve."""
    n = 1
    while n < max(nx, ny):
        n *= 2
    x, y = np.meshgrid(np.arange(nx), np.arange(ny))
    x, y = x.reshape(-1).astype(np.int64), y.reshape(-1).astype(np.int64)
    d = np.zeros_like(x)
    s = n // 2
    while s:
        rx, ry = (x & s) > 0, (y & s) > 0
        d += s * s * ((3 * rx) ^ ry)
        flip = ~ry & rx
        x, y = np.where(flip, n - 1 - x, x), np.where(flip, n - 1 - y, y)
        x, y = np.where(~ry, y, x), np.where(~ry, x, y)
        s //= 2
    return torch.from_numpy(np.argsort(d)).to(_DEV)


def _wavefield(g, ns, nr):
    """D (ns x nr): a corner of F diag(sigma e^{i phi}) P F diag(psi), sigma from 1 to 1e-3."""
    n = max(ns, nr)
    u = torch.rand(2, n, device=_DEV, generator=g)
    one = torch.ones(n, device=_DEV)
    m = torch.fft.fft(torch.diag(torch.polar(one, 2 * math.pi * u[0])), dim=0)
    sigma = torch.logspace(0, -3, n, device=_DEV)
    m = m[torch.randperm(n, device=_DEV, generator=g)] * torch.polar(sigma, 2 * math.pi * u[1])[:, None]
    return (torch.fft.fft(m, dim=0)[:ns, :nr] / n).contiguous()


def _data(c, g):
    """D, U (ns x nr, natural receiver order) of a planted X."""
    nr, ns = c["nx"] * c["ny"], c["ns"]
    D = _wavefield(g, ns, nr)
    order = _hilbert(c["nx"], c["ny"])
    Uh = D[:, order] @ _assemble(c, _theta(c, g))
    U = torch.empty_like(D)
    U[:, order] = Uh
    e = _randn(g, ns, nr)
    U += e * (torch.linalg.norm(U) / torch.linalg.norm(e) * 10 ** (-c["snr"] / 20))
    return D, U


def _desc(c):
    t = _tiles(c)
    return T.desc(c["nx"] * c["ny"], c["ns"], c["tile"], rank=c["rank"], nx=c["nx"], ny=c["ny"],
                  diag_mode=_DIAG[c["diag"]], precision=_PREC[c["prec"]], tiles=t if c["tile2"] else None,
                  reciprocity=T.TLR_RECIP_NONE if c["general"] else T.TLR_RECIP_SYMMETRIC)


class _State:
    """A prepared case; destroys its handle when it goes."""

    def __init__(self, case):
        self.case, self.handle, self.stream = case, None, None

    def __del__(self):
        if self.handle is not None:
            T.tlr_mdd_destroy(self.handle)
            self.handle = None


def _symmetric(c, g):
    """What the benchmark solver leaves: a symmetric planted X in a little noise."""
    X = _assemble(c, _theta(c, g))
    e = _randn(g, *X.shape)
    return (X + (1e-3 * torch.linalg.norm(X) / torch.linalg.norm(e)) * (e + e.T)).contiguous()


def prepare(case, seed):
    g = torch.Generator(device=_DEV).manual_seed(int(seed))
    s = _State(case)
    kind = case["kind"]
    if kind == "stack":
        s.x = torch.randn(case["ntr"], case["nt"], device=_DEV, generator=g)
        s.xw = torch.empty((case["nf"], case["ntr"]), dtype=torch.complex64, device=_DEV)
        s.y = torch.empty_like(s.x)
        return s
    nr, ns = case["nx"] * case["ny"], case["ns"]
    D, U = _data(case, g)
    s.desc = _desc(case)
    n = T.tlr_mdd_theta_size(s.desc)
    if kind == "create":
        s.D, s.U = D, U
        s.Dt = torch.empty((nr, ns), dtype=torch.complex64, device=_DEV)
        s.Ut = torch.empty_like(s.Dt)
        return s
    if kind == "solve":
        s.stream = torch.cuda.Stream()     # a solve on a stream of its own is recorded and replayed
        s.stream.wait_stream(torch.cuda.current_stream())
        torch.cuda.synchronize()
    s.handle = T.tlr_mdd_create(s.desc, D, U, s.stream)
    if kind == "solve":
        s.start = 0.1 * _theta(case, g)
        s.theta = torch.empty_like(s.start)
        s.X = torch.empty((nr, nr), dtype=torch.complex64, device=_DEV)
        s.opts = T.solve_opts(stages=case["stages"])
    elif kind in ("grad", "apply"):
        s.theta = _theta(case, g)
        if kind == "grad":
            s.grad = torch.empty_like(s.theta)
        else:
            s.Y = torch.empty((nr, ns), dtype=torch.complex64, device=_DEV)
    elif kind == "adjoint":
        s.V = _randn(g, nr, ns)
        s.G = torch.empty((nr, nr), dtype=torch.complex64, device=_DEV)
    elif kind == "benchmark":
        s.X = torch.empty((nr, nr), dtype=torch.complex64, device=_DEV)
    elif kind == "warm":
        s.Xb = _symmetric(case, g)
        s.theta = torch.empty(n, dtype=torch.complex64, device=_DEV)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "solve":
        with torch.cuda.stream(s.stream):
            s.theta.copy_(s.start)
            st = T.tlr_mdd_solve(s.handle, s.theta, s.opts)
            T.tlr_mdd_unpermute_dense(s.handle, s.theta, s.X)
        return {"theta": s.theta, "X": s.X, "f0": st.f0, "iters": st.iters,
                "f": torch.tensor(list(st.f_hist)[:st.n_hist], dtype=torch.float32)}
    if kind == "grad":
        return {"f": T.tlr_mdd_grad(s.handle, s.theta, s.grad), "grad": s.grad}
    if kind == "apply":
        T.tlr_mdd_apply(s.handle, s.theta, s.Y)
        return s.Y
    if kind == "adjoint":
        T.tlr_mdd_adjoint(s.handle, s.V, s.G)
        return s.G
    if kind == "create":
        h = T.tlr_mdd_create(s.desc, s.D, s.U)
        perm, alpha = T.tlr_mdd_get_data(h, c["nx"] * c["ny"], s.Dt, s.Ut)
        T.tlr_mdd_destroy(h)
        return {"perm": np.asarray(perm), "alpha": alpha, "D": s.Dt, "U": s.Ut}
    if kind == "benchmark":
        st = T.tlr_mdd_benchmark_solve(s.handle, 0.01, 20, 0.0, s.X)
        return {"X": s.X, "iters": st.iters}
    if kind == "warm":
        ranks, entries, v0 = (0, 0, 0.0)
        if not c["tile2"]:
            ranks, entries, v0 = T.tlr_mdd_tile_ranks(s.Xb, c["nx"] * c["ny"], c["tile"], 0.01)
        T.tlr_mdd_warm_start(s.handle, s.Xb, s.theta)
        return {"ranks": np.asarray(ranks), "entries": entries, "v0": v0, "theta": s.theta}
    T.tlr_mdd_time_to_freq(s.x, c["ntr"], c["nt"], c["f0"], c["nf"], s.xw)
    T.tlr_mdd_freq_to_time(s.xw, c["ntr"], c["nt"], c["f0"], c["nf"], s.y)
    return {"stack": s.xw, "traces": s.y}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    c = case
    if c["kind"] == "stack":
        ntr, nt, nf = c["ntr"], c["nt"], c["nf"]
        return {"bytes": 2.0 * ntr * (4 * nt + 8 * nf), "flops": 2 * 2.5 * ntr * nt * math.log2(max(2, nt))}
    nr, ns = c["nx"] * c["ny"], c["ns"]
    panel = 8.0 * nr * ns
    theta = sum(r * k for _, _, _, r, k in _blocks(c))
    low = sum(r * k for kind, _, _, r, k in _blocks(c) if kind != "Z")
    z = theta - low
    kind = c["kind"]
    # per complex factor entry and source: compress and expand 8 flops each; dense diagonal entries are used once
    forward = ns * (8.0 * (1 if c["general"] else 2) * low + 8.0 * z)
    if kind == "apply":
        return {"bytes": 2 * panel + 8 * theta, "flops": forward}
    grad = forward + ns * (8.0 * (2 if c["general"] else 3) * low + 8.0 * z)
    if kind == "grad":
        return {"bytes": 2 * panel + 16 * theta, "flops": grad}
    if kind == "solve":
        per = ns * (8.0 * (4 if c["general"] else 7) * low + 16.0 * z)
        return {"bytes": 2 * panel + 16 * theta + 8.0 * nr * nr, "flops": grad + 10 * c["stages"] * per}
    if kind == "adjoint":
        return {"bytes": 2 * panel + 8.0 * nr * nr, "flops": 8.0 * nr * nr * ns}
    if kind == "create":
        return {"bytes": 4 * panel, "flops": 2.0 * nr * ns}
    if kind == "benchmark":
        return {"bytes": 2 * panel + 8.0 * nr * nr, "flops": 16.0 * nr * nr * ns + 20 * 8.0 * nr ** 3}
    # warm: singular values of the lower tiles, then singular vectors too (about 8/3 and 20 real d^3 flops, complex)
    tiles = [(d, e) for i, d in enumerate(_tiles(c)) for e in _tiles(c)[:i + 1]]
    return {"bytes": 2 * 4.0 * nr * nr + 8 * theta, "flops": sum(4 * (8 / 3 + 20) * d * e * min(d, e) for d, e in tiles)}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _panels(c, D, U):
    order = _hilbert(c["nx"], c["ny"])
    D, U = D.to(torch.complex128), U.to(torch.complex128)
    alpha = float(D.abs().max())
    return D[:, order].T / alpha, U[:, order].T / alpha, alpha, order


def _forward(c, f, D):
    rows = _rows(c)
    Y = torch.zeros_like(D)
    for i, r in enumerate(rows):
        if ("Z", i, i) in f:
            Z = f["Z", i, i]
            Y[r] += (Z.T if c["general"] else 0.5 * (Z + Z.T)) @ D[r]
        elif c["general"]:
            Y[r] += f["QR", i, i] @ (f["QL", i, i].T @ D[r])
        else:
            Y[r] += f["Q", i, i] @ (f["Q", i, i].T @ D[r])
    for i, j in _pairs(c):
        L, R = f["L", i, j], f["R", i, j]
        Y[rows[j]] += R @ (L.T @ D[rows[i]])
        if not c["general"]:
            Y[rows[i]] += L @ (R.T @ D[rows[j]])
    return Y


def _gradient(c, f, D, R):
    """Blocks of the gradient of 0.5 ||Y - U||^2, stacked as theta is; R = Y - U."""
    rows, got = _rows(c), {}
    cD = D.conj()
    for i, r in enumerate(rows):
        if ("Z", i, i) in f:
            G = R[r] @ cD[r].T
            got["Z", i, i] = G.T if c["general"] else 0.5 * (G + G.T)
        elif c["general"]:
            QL, QR = f["QL", i, i].conj(), f["QR", i, i].conj()
            got["QL", i, i] = cD[r] @ (R[r].T @ QR)
            got["QR", i, i] = R[r] @ (cD[r].T @ QL)
        else:
            Q = f["Q", i, i].conj()
            got["Q", i, i] = R[r] @ (cD[r].T @ Q) + cD[r] @ (R[r].T @ Q)
    for i, j in _pairs(c):
        L, Rf, ri, rj = f["L", i, j].conj(), f["R", i, j].conj(), rows[i], rows[j]
        got["L", i, j] = cD[ri] @ (R[rj].T @ Rf)
        got["R", i, j] = R[rj] @ (cD[ri].T @ L)
        if not c["general"]:
            got["L", i, j] += R[ri] @ (cD[rj].T @ Rf)
            got["R", i, j] += cD[rj] @ (R[ri].T @ L)
    return torch.cat([got[kind, i, j].reshape(-1) for kind, i, j, _, _ in _blocks(c)])


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "solve":
        return None      # 10 to 30 iterations: each rounds what the next one starts from
    g = torch.Generator(device=_DEV).manual_seed(int(seed))
    if kind == "stack":
        x = torch.randn(c["ntr"], c["nt"], device=_DEV, generator=g)
        w = torch.fft.rfft(x.double(), dim=1)[:, c["f0"]:c["f0"] + c["nf"]]
        full = torch.zeros((c["ntr"], c["nt"] // 2 + 1), dtype=torch.complex128, device=_DEV)
        full[:, c["f0"]:c["f0"] + c["nf"]] = w
        return {"stack": w.T.contiguous(), "traces": torch.fft.irfft(full, n=c["nt"], dim=1)}
    D, U = _data(c, g)
    Dt, Ut, alpha, order = _panels(c, D, U)
    if kind == "create":
        return {"perm": order.cpu(), "alpha": alpha, "D": Dt, "U": Ut}
    if kind in ("grad", "apply"):
        f = _factors(c, _theta(c, g).to(torch.complex128))
        Y = _forward(c, f, Dt)
        if kind == "apply":
            return Y
        Y -= Ut
        return {"f": 0.5 * float(torch.linalg.norm(Y)) ** 2, "grad": _gradient(c, f, Dt, Y)}
    if kind == "adjoint":
        return _randn(g, *Dt.shape).to(torch.complex128) @ Dt.conj().T
    if kind == "benchmark":
        def sym(a):
            return 0.5 * (a + a.T)
        G, r = Dt.conj() @ Dt.T, sym(Dt.conj() @ Ut.T)
        x, p = torch.zeros_like(r), r.clone()
        rr = float(torch.linalg.norm(r)) ** 2
        for _ in range(20):
            a = sym(G @ p) + 0.02 * p
            step = rr / float((p.conj() * a).sum().real)
            x += step * p
            r -= step * a
            new = float(torch.linalg.norm(r)) ** 2
            p = r + (new / rr) * p
            rr = new
        return {"X": x, "iters": None}
    # warm: the largest singular value; singular vectors are defined up to a phase
    X, rows = _symmetric(c, g).to(torch.complex128), _rows(c)
    v0 = None if c["tile2"] else max(float(torch.linalg.matrix_norm(X[rows[i], rows[j]], 2))
                                     for i in range(len(rows)) for j in range(i + 1))
    return {"ranks": None, "entries": None, "v0": v0, "theta": None}
