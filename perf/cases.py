"""What a user of this framework has it compute, as timed cases.

A pass is one simulation through the public classes of
paper_1505_02037_gb300.lbnr: initial fields from pinned host memory, a number
of steps, and the corrected moments (or a batch's distributions) read back.
Each pass starts from the same initial fields, as the steps of a parameter
study do, so passes can be repeated without running into the scheme's own
growth (the linear amplification of a step is 1.0029 at tau = 4.5).

The results arrive as float64 whatever the storage. A run whose state is held
in 32 or 16 bits hands them on to its post-processing on the GPU in that type.

exact() evolves the same initial fields in float64 with plain torch.
"""
import math

import numpy as np
import torch

from paper_1505_02037_gb300 import autotune, lbnr

Q_OF = {1: 3, 2: 9, 3: 19}
BYTES = {"f64": 8, "f32": 4, "dev_f32": 4, "dev_bf16": 2, "dev_f16": 2}
KEEP = {"f32": torch.float32, "dev_f32": torch.float32, "dev_bf16": torch.bfloat16,
        "dev_f16": torch.float16}
SLICING = {"geodesic": 0, "harmonic": 1, "1+log": 2}
STREAMING = {"auto": 0, "pingpong": 1, "aa": 2}
SHIFT = (0.05, 0.02, -0.02)


def _lattice(name, vset, shape, storage, steps, **more):
    nx, ny, nz = (tuple(shape) + (1, 1))[:3]
    c = dict(name=name, kind="lattice", vset=vset, nx=nx, ny=ny, nz=nz, storage=storage,
             steps=steps, checks=1, tau=4.5, amplitude=0.1, direction="x", mix=0.05,
             slicing="harmonic", streaming="auto", deriv="sync", shift="none", monitor=False,
             tuned=False)
    c.update(more)
    return c


def listed():
    return [
        # the paper's 1D gauge wave, 200 cells to t = 10: a few kilobytes a step, so
        # latency and launches are everything
        _lattice("wave1d-200-f64", 1, (200,), "f64", 2000, mix=0.001),
        # one line of the paper's tau sweep (reproduce.py): 800 cells of D2Q9 and four
        # rows, the moments read every 10 steps
        _lattice("sweep2d-800x4-f64", 2, (800, 4), "f64", 100, checks=10, tau=3.0,
                 amplitude=1e-3),
        # a reference run in FP64 with the constraint monitor every 10 steps
        _lattice("monitor3d-64-f64", 3, (64, 64, 64), "f64", 40, checks=4, direction="xyz",
                 monitor=True),
        # a 2D run of ordinary size, FP32, a lattice of no round size
        _lattice("wave2d-1000-f32", 2, (1000, 1000), "f32", 200, direction="xy"),
        # the quick start of the README: 128^3, FP32, 100 steps, defaults everywhere
        _lattice("quickstart3d-128-f32", 3, (128, 128, 128), "f32", 100),
        # the headline run, set up as bench.py does (launch form from the autotuner)
        _lattice("wave3d-256-f32", 3, (256, 256, 256), "f32", 100, tuned=True),
        # the same lattice at half the bytes, for qualitative scans
        _lattice("wave3d-256-dev_f16", 3, (256, 256, 256), "dev_f16", 100, amplitude=0.01,
                 tuned=True),
        # a ragged box in place (one buffer), 1+log slicing, FP32 deviations: the storage
        # that keeps the FP64 error
        _lattice("ragged3d-149x101x67-dev_f32-aa", 3, (149, 101, 67), "dev_f32", 100,
                 slicing="1+log", streaming="aa"),
        # lagged derivatives: one kernel a step
        _lattice("lag3d-160-dev_f32", 3, (160, 160, 160), "dev_f32", 100, direction="xyz",
                 deriv="lag"),
        # prescribed shift, constant part and static shear field
        _lattice("shift3d-128-f32", 3, (128, 128, 128), "f32", 100, amplitude=0.01,
                 shift="field"),
        # the comparison scheme with A and D evolved (37 fields)
        dict(name="ad3d-96-f32", kind="ad", vset=3, nx=96, ny=96, nz=96, storage="f32",
             steps=150, tau=4.5, amplitude=0.1, direction="x", mix=0.05, slicing="harmonic"),
        # a parameter scan: 32 uneven 1D and 2D runs in one launch
        dict(name="ensemble-32-dev_f32", kind="batch", runs=32, n1_lo=64, n1_hi=4096, n2_lo=64,
             n2_hi=192, storage="dev_f32", deriv="sync", crossings=6, layout=150502037),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: set, size, storage, streaming and options as users mix them."""
    kind = rng.choice(["1d", "2d", "3d", "3d", "3d", "3d", "ad", "batch"])
    tau = rng.uniform(4.0, 5.5)
    slicing = rng.choice(["harmonic", "harmonic", "harmonic", "1+log", "geodesic"])
    if kind == "batch":
        lo = rng.randint(16, 64)
        return dict(kind="batch", runs=rng.randint(8, 32), n1_lo=rng.randint(32, 128),
                    n1_hi=rng.randint(500, 4096), n2_lo=lo, n2_hi=lo + rng.randint(32, 128),
                    storage=rng.choice(["dev_f32", "dev_f32", "f64"]),
                    deriv=rng.choice(["sync", "sync", "lag"]), crossings=rng.randint(1, 4),
                    layout=rng.randint(1, 1 << 30))
    if kind == "ad":
        side = [_log_int(rng, 16, 112) for _ in range(3)]
        cells = side[0] * side[1] * side[2]
        return dict(kind="ad", vset=3, nx=side[0], ny=side[1], nz=side[2],
                    storage=rng.choice(["f32", "f32", "f64"]) if cells < 100000 else "f32",
                    steps=rng.randint(20, 120), tau=tau, amplitude=0.05, direction="x", mix=0.02,
                    slicing=slicing)
    storage = rng.choice(["f64", "f32", "f32", "dev_f32", "dev_f32", "dev_f16", "dev_bf16"])
    if kind == "1d":
        # fine lattices: FP64, or the deviations that keep its error
        vset, shape, storage = 1, (_log_int(rng, 64, 4096),), rng.choice(["f64", "f64", "dev_f32"])
    elif kind == "2d":
        vset, shape = 2, (_log_int(rng, 32, 2000), _log_int(rng, 4, 2000))
    else:
        vset, shape = 3, tuple(_log_int(rng, 8, 240) for _ in range(3))
    cells = int(np.prod(shape))
    work = cells * Q_OF[vset] * (8.0 if storage == "f64" else 1.0)
    # at most a crossing and a half of the box along x: later the scheme's own growth
    # would carry rounding into the results
    steps = max(10, min(int(1.5 * shape[0]), 1000 if vset == 1 else 200, int(2e10 / work)))
    shift = rng.choice(["none", "none", "none", "constant", "field"])
    if storage.endswith("16"):
        shift = "none"
    case = _lattice("", vset, shape, storage, steps, tau=tau, amplitude=rng.choice([0.01, 0.05]),
                    mix=0.001 if steps > shape[0] else 0.02, slicing=slicing,
                    streaming=rng.choice(["auto", "auto", "aa"]),
                    deriv=rng.choice(["sync", "sync", "lag"]), shift=shift,
                    monitor=storage == "f64" and cells < 300000,
                    tuned=rng.random() < 0.3)
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _fields(shape, amplitude, direction, mix, seed):
    """[16][nz][ny][nx] on the GPU, float64: the gauge wave of seeded amplitude
    and phase on the unit-length box, plus one low Fourier mode of amplitude
    mix * amplitude in each field, so that every term of the equations is live."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = shape
    dx = 1.0 / nx
    dev = "cuda"
    x = (torch.arange(nx, device=dev, dtype=torch.float64) + 0.5) * dx
    y = (torch.arange(ny, device=dev, dtype=torch.float64) + 0.5) * dx
    z = (torch.arange(nz, device=dev, dtype=torch.float64) + 0.5) * dx
    axes = (x[None, None, :], y[None, :, None], z[:, None, None])
    box = (nx * dx, ny * dx, nz * dx)
    n = {"x": (1, 0, 0), "xy": (1, 1, 0), "xyz": (1, 1, 1)}[direction]
    norm = math.sqrt(sum(n))
    n = [v / norm for v in n]
    d = 1.0 / norm  # wavelength: periodic on the box
    A = amplitude * rng.uniform(0.8, 1.0)
    ph = 2 * math.pi / d * (n[0] * axes[0] + n[1] * axes[1] + n[2] * axes[2]) + rng.uniform(0, 6.28)
    H = (1 - A * torch.sin(ph)).expand(nz, ny, nx)
    Knn = -(math.pi * A / d) * torch.cos(ph).expand(nz, ny, nx) / H.sqrt()
    out = torch.zeros((16, nz, ny, nx), dtype=torch.float64, device=dev)
    out[0] = H.sqrt()
    for q, (i, j) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
        out[1 + q] = (1.0 if i == j else 0.0) + (H - 1) * (n[i] * n[j])
        out[7 + q] = Knn * (n[i] * n[j])
    live = [a for a in range(3) if shape[a] > 1]
    for F in range(16):
        k = [0, 0, 0]
        for a in live:
            k[a] = int(rng.integers(-1, 2))
        if not any(k):
            k[live[0]] = 1
        arg = 2 * math.pi * sum(k[a] * axes[a] / box[a] for a in range(3)) + rng.uniform(0, 6.28)
        out[F] += mix * amplitude * rng.uniform(0.5, 1.0) * torch.sin(arg)
    return out


def _shift_field(shape, v0=0.02):
    """A divergence-free shear: each component varies across its own direction."""
    nx, ny, nz = shape
    g = np.meshgrid(*((np.arange(m) + 0.5) / m for m in (nz, ny, nx)), indexing="ij")
    return v0 * np.sin(2 * math.pi * np.stack([g[1], g[0], g[2]]))


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


def _shape(case):
    return (case["nx"], case["ny"], case["nz"])


def _runs(case):
    """The scan's runs: sizes, relaxation times and amplitudes from its layout number."""
    rng = np.random.default_rng(case["layout"])
    runs = []
    for r in range(case["runs"]):
        vset = 1 + r % 2
        lo, hi = (case["n1_lo"], case["n1_hi"]) if vset == 1 else (case["n2_lo"], case["n2_hi"])
        N = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        runs.append(dict(vset=vset, shape=(N, 1 if vset == 1 else N, 1), dx=1.0 / N,
                         tau=float(rng.uniform(4.5, 6.5)), slicing=1,
                         amplitude=float(math.exp(rng.uniform(math.log(1e-3), math.log(0.1)))),
                         direction="xy" if vset == 2 and r % 4 == 1 else "x",
                         steps=min(case["crossings"] * N, 1200)))
    return runs


def _shifts(case):
    return {"none": (None, False), "constant": (SHIFT, False), "field": (SHIFT, True)}[case["shift"]]


def prepare(case, seed):
    if case["kind"] == "batch":
        runs = _runs(case)
        fields = [_fields(r["shape"], r["amplitude"], r["direction"], 0.001, seed + 7919 * i)
                  .reshape(16, -1).cpu().numpy() for i, r in enumerate(runs)]
        batch = lbnr.Batch(runs, storage=case["storage"], deriv_mode=case["deriv"])
        return dict(case=case, batch=batch, fields=fields)
    shape = _shape(case)
    fields = _fields(shape, case["amplitude"], case["direction"], case["mix"], seed)
    if case["kind"] == "ad":
        lat = lbnr.ADLattice(case["vset"], shape, case["tau"], 1.0 / shape[0],
                             slicing=SLICING[case["slicing"]], storage=case["storage"])
        return dict(case=case, lat=lat, fields=fields.reshape(16, -1).cpu().numpy())
    lat = lbnr.Lattice(case["vset"], shape, case["tau"], 1.0 / shape[0],
                       slicing=SLICING[case["slicing"]], storage=case["storage"],
                       streaming=STREAMING[case["streaming"]], deriv_mode=case["deriv"])
    beta, field = _shifts(case)
    if beta is not None:
        lat.set_shift(beta)
    if field:
        lat.set_shift_field(_shift_field(shape))
    state = dict(case=case, lat=lat, fields=_pinned(fields.reshape(16, -1)),
                 out=torch.empty((case["checks"], 16, lat.cells), dtype=torch.float64,
                                 pin_memory=True))
    del fields
    if case["tuned"]:
        lat.init(state["fields"])
        autotune.tune(lat)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        for i, f in enumerate(state["fields"]):
            b.init(i, f)
        b.run()
        b.check()
        got = [torch.from_numpy(b.distributions(i)) for i in range(len(b))]
        return got if case["storage"] == "f64" else [g.float() for g in got]
    lat = state["lat"]
    lat.init(state["fields"])
    if case["kind"] == "ad":
        lat.step(case["steps"])
        m = torch.from_numpy(lat.moments())
        return m if case["storage"] == "f64" else m.float()
    out, monitor = state["out"], []
    for k in range(case["checks"]):
        lat.step(case["steps"] // case["checks"])
        lat.moments(out[k])
        if case["monitor"]:
            monitor.append(torch.from_numpy(lat.constraints()))
    if case["storage"] != "f64":
        return out.to("cuda", non_blocking=True).to(KEEP[case["storage"]])
    return [out, torch.stack(monitor)] if monitor else out


def work(case):
    """Bytes: initial fields read, the state written, read and written again each
    step, the results written. Operations: sums and relaxation of every value,
    and about 700 for the sources and fluxes of a cell."""
    if case["kind"] == "batch":
        b = fl = 0.0
        s = BYTES[case["storage"]]
        for r in _runs(case):
            cells, Q = r["shape"][0] * r["shape"][1], Q_OF[r["vset"]]
            b += cells * (128 + 16 * Q * (s * (2 * r["steps"] + 2) + 8))
            fl += cells * r["steps"] * (16 * Q * 4 + 700.0)
        return {"bytes": b, "flops": fl}
    nf = 37 if case["kind"] == "ad" else 16
    cells, Q = case["nx"] * case["ny"] * case["nz"], Q_OF[case["vset"]]
    n, s, checks = case["steps"], BYTES[case["storage"]], case.get("checks", 1)
    return {"bytes": cells * (128.0 + nf * Q * s * (2 * n + 1 + checks) + nf * 8 * checks),
            "flops": float(cells * n * (nf * Q * 4 + 700))}


# ---------------------------------------------------------------------------
# The same runs in float64, plain torch
# ---------------------------------------------------------------------------
C19 = ("0 + - 0 0 0 0 + - + - + - + - 0 0 0 0", "0 0 0 + - 0 0 - + + - 0 0 0 0 + - + -",
       "0 0 0 0 0 + - 0 0 0 0 - + + - - + + -")
C9 = ("0 + - 0 0 + - + -", "0 0 0 + - - + + -", "0 0 0 0 0 0 0 0 0")
C3 = ("0 + -", "0 0 0", "0 0 0")
SYM = ((0, 1, 2), (1, 3, 4), (2, 4, 5))


def _velocities(vset):
    rows = {1: C3, 2: C9, 3: C19}[vset]
    c = [tuple({"0": 0, "+": 1, "-": -1}[r.split()[l]] for r in rows)
         for l in range(len(rows[0].split()))]
    w = {1: (2 / 3, 1 / 6, None), 2: (4 / 9, 1 / 9, 1 / 36), 3: (1 / 3, 1 / 18, 1 / 36)}[vset]
    return c, [w[sum(abs(v) for v in cl)] for cl in c]


def _full(s):
    """[6][n] to the symmetric [3][3][n]."""
    return s[[q for row in SYM for q in row]].reshape(3, 3, -1)


def _six(m):
    """[3][3][n] to its six pairs."""
    return torch.stack([m[0, 0], m[0, 1], m[0, 2], m[1, 1], m[1, 2], m[2, 2]])


def _dot(a, b, dim):
    return (a * b).sum(dim)


def _inverse(g):
    c = torch.stack([torch.linalg.cross(g[(i + 1) % 3], g[(i + 2) % 3], dim=0) for i in range(3)])
    return c / _dot(g[0], c[0], 0)


def _point(m, A, D, slicing, B=None, beta=None):
    """Sources S[16][n] of the fields m[16][n] with A[3][n], D[3][3][3][n] = D_kij."""
    al, g, K, V = m[0], _full(m[1:7]), _full(m[7:13]), m[13:16]
    gi = _inverse(g)
    Km = _dot(gi[:, :, None], K[None], 1)                     # K^i_j
    trK = Km[0, 0] + Km[1, 1] + Km[2, 2]
    trK2 = (Km * Km.transpose(0, 1)).sum((0, 1))
    Dl = _dot(D[:, :, :, None], gi[None, None], 2)            # D_ki^r
    Du = _dot(gi[:, :, None, None], D[None], 1)               # D^k_ij
    t1 = torch.stack([sum(Dl[k, r, r] for r in range(3)) for k in range(3)])   # D_kr^r
    t2 = torch.stack([sum(Dl[r, k, r] for r in range(3)) for k in range(3)])   # D^r_rk
    up = lambda v: _dot(gi, v[None], 1)  # noqa: E731
    Au, Vu, t1u, Dkk = up(A), up(V), up(t1), up(t2)
    low = Dl.permute(2, 0, 1, 3)                              # [k][i][j] = D_ij^k
    G = low + low.transpose(1, 2) - Du                        # Gamma^k_ij
    Gc = torch.stack([sum(G[k, k, r] for k in range(3)) for r in range(3)])
    Duu = _dot(gi[None, :, :, None], Dl[:, None], 2)          # D_k^{rs}
    bracket = (-(Duu * G).sum((0, 1, 2)) + _dot(t1, t1u, 0) - 2 * _dot(Vu, A, 0) + trK2
               - trK * trK)
    M = torch.stack([torch.stack([sum(Dl[i, k, r] * Dl[r, j, k] for k in range(3)
                                      for r in range(3)) for j in range(3)]) for i in range(3)])
    GG = torch.stack([torch.stack([sum(G[k, r, i] * G[r, k, j] for k in range(3)
                                       for r in range(3)) for j in range(3)]) for i in range(3)])
    S = -2 * _dot(K[:, :, None], Km[None], 1) + trK * K + 2 * (M + M.transpose(0, 1)) - GG
    S = S + (Gc[:, None, None] * G).sum(0)
    e = 2 * Dkk - Au
    X = _dot(D, e[None, None], 2)                             # D_ijr e^r
    S = S - X - X.transpose(0, 1) - (Vu[:, None, None] * D).sum(0)
    h = V - 0.5 * t1
    S = S + A[:, None] * h[None] + A[None] * h[:, None] + 0.25 * g * bracket
    out = torch.empty_like(m)
    out[7:13] = al * _six(S)
    Om = _dot(A[:, None], Km, 0) - trK * A - _dot(Km, (t1 - 2 * t2)[:, None], 0)
    Om = Om + ((Dl - 2 * Dl.transpose(0, 1)) * Km[None]).sum((1, 2))
    out[13:16] = al * Om
    Qs = (torch.zeros_like(al), trK, trK / al)[slicing]
    out[0] = -al * al * Qs
    out[1:7] = -2 * al * m[7:13]
    if beta is not None:
        out[0] += al * _dot(beta, A, 0)
        out[1:7] += 2 * _six((beta[:, None, None] * D).sum(0))
    if B is not None:                                         # B[k][i] = d_k beta^i / 2
        Bl = _dot(B[:, :, None], g[None], 1)
        Bu = _dot(gi[:, :, None], Bl[None], 1)                # B^r_s
        trB = B[0, 0] + B[1, 1] + B[2, 2]
        out[1:7] += 2 * _six(Bl + Bl.transpose(0, 1))
        KB = _dot(K[:, None], B[None], 2)                     # K_ir B_j^r
        out[7:13] += 2 * _six(KB + KB.transpose(0, 1) - K * trB)
        om = _dot(B, V[None], 1) - trB * V
        om = om + (Dl.transpose(0, 1) * Bu[None]).sum((1, 2)) - _dot(t2[:, None], Bu, 0)
        out[13:16] += 2 * om
    return out


def _fluxes(m, A, D, B=None, beta=None):
    """Fluxes along each axis: K [3][6][n], V [3][3][n] (zero without a shift)."""
    al, g, K, V = m[0], _full(m[1:7]), m[7:13], m[13:16]
    gi = _inverse(g)
    t1 = (gi[None] * D).sum((1, 2))
    e = 0.5 * (A + 2 * V - t1)
    Vu = _dot(gi, V[None], 1)
    lam = _dot(gi[:, :, None, None], D[None], 1) - 0.5 * Vu[:, None, None] * g[None]
    for k in range(3):
        lam[k, k] += e
        lam[k, :, k] += e
    FK = al * torch.stack([_six(lam[k]) for k in range(3)])
    FV = torch.zeros((3,) + tuple(V.shape), dtype=V.dtype, device=V.device)
    if beta is not None:
        FK -= beta[:, None] * K[None]
        FV -= beta[:, None] * V[None]
    if B is not None:
        Bl = _dot(B[:, :, None], g[None], 1)
        FV += _dot(gi[:, :, None], Bl[None], 1) - B.transpose(0, 1)  # B^k_i - B_i^k
    return FK, FV


class _Exact:
    """The 16- or 37-field scheme on one periodic lattice, float64."""

    CHUNK = 1 << 19

    def __init__(self, vset, shape, tau, slicing, dev, deriv="sync", shift="none", ad=False):
        self.c, self.w = _velocities(vset)
        self.dim, self.shape, self.tau, self.slicing = vset, shape, tau, slicing
        self.dx, self.dev, self.lag, self.ad = 1.0 / shape[0], dev, deriv == "lag", ad
        self.nf = 37 if ad else 16
        self.beta = self.B = None
        if shift != "none":
            nx, ny, nz = shape
            b = torch.tensor(SHIFT, dtype=torch.float64, device=dev)[:, None].repeat(1, nx * ny * nz)
            if shift == "field":
                b = b + torch.from_numpy(_shift_field(shape)).to(dev).reshape(3, -1)
                self.B = torch.stack([self._diff(b, k) / 2 for k in range(3)])
            self.beta = b

    def _diff(self, v, k):
        """Central difference along axis k (zero where the set has no velocity)."""
        nx, ny, nz = self.shape
        if k >= self.dim:
            return torch.zeros_like(v)
        t = v.reshape(-1, nz, ny, nx)
        return ((t.roll(-1, 3 - k) - t.roll(1, 3 - k)) / (2 * self.dx)).reshape(v.shape)

    def _derivs(self, m7):
        la = m7[0].log()
        A = torch.stack([self._diff(la, k) for k in range(3)])
        D = torch.stack([self._diff(m7[1:7], k) / 2 for k in range(3)])
        return A, D

    def _pieces(self, rt, A, D, body):
        n = rt.shape[1]
        for i in range(0, n, self.CHUNK):
            s = slice(i, min(n, i + self.CHUNK))
            if self.ad:
                a, d = rt[16:19, s], rt[19:37, s].reshape(3, 6, -1)
            else:
                a, d = A[:, s], D[:, :, s]
            d = torch.stack([_full(d[k]) for k in range(3)])
            b = None if self.beta is None else self.beta[:, s]
            B = None if self.B is None else self.B[:, :, s]
            body(s, rt[:16, s], a, d, B, b)

    def _equilibrium(self, rho, A, D, F):
        """Fluxes of every field into F[3][nf][n] at rho."""
        def body(s, m, a, d, B, b):
            FK, FV = _fluxes(m, a, d, B, b)
            F[:, 7:13, s] = FK
            F[:, 13:16, s] = FV
            if self.ad:
                gi = _inverse(_full(m[1:7]))
                trK = (gi * _full(m[7:13])).sum((0, 1))
                aQ = (torch.zeros_like(trK), m[0] * trK, trK)[self.slicing]
                for k in range(3):
                    F[k, 16 + k, s] = aQ
                    F[k, 19 + 6 * k:25 + 6 * k, s] = m[0] * m[7:13]
        self._pieces(rho, A, D, body)

    def _sources(self, rt, A, D):
        S = torch.zeros_like(rt)

        def body(s, m, a, d, B, b):
            S[:16, s] = _point(m, a, d, self.slicing, B, b)
        self._pieces(rt, A, D, body)
        return S

    def init(self, fields):
        r = fields.reshape(16, -1)
        A, D = self._derivs(r)
        if self.ad:
            r = torch.cat([r, A, D.reshape(18, -1)])
        S = self._sources(r, A, D)
        F = torch.zeros((3,) + tuple(r.shape), dtype=r.dtype, device=r.device)
        self._equilibrium(r, A, D, F)
        self.f = torch.empty((len(self.w),) + tuple(r.shape), dtype=r.dtype, device=r.device)
        for l, (c, w) in enumerate(zip(self.c, self.w)):
            self.f[l] = w * (r + 3 * sum(c[k] * F[k] for k in range(3)) - self.dx / 2 * S)
        self.prev = r[:7].clone() if self.lag else None
        self.F = F

    def _macro(self):
        rt = self.f.sum(0)
        A = D = None
        if not self.ad:
            A, D = self._derivs(self.prev if self.lag else rt)
        S = self._sources(rt, A, D)
        return rt + self.dx / 2 * S, S, A, D

    def moments(self):
        return self._macro()[0]

    def step(self):
        rho, S, A, D = self._macro()
        om, F = 1 / self.tau, self.F
        self._equilibrium(rho, A, D, F)
        base = om * rho + self.dx * (1 - om / 2) * S
        nx, ny, nz = self.shape
        for l, (c, w) in enumerate(zip(self.c, self.w)):
            v = (1 - om) * self.f[l] + w * (base + 3 * om * sum(c[k] * F[k] for k in range(3) if c[k]))
            self.f[l] = v.reshape(-1, nz, ny, nx).roll((c[2], c[1], c[0]), (1, 2, 3)).reshape(v.shape)
        if self.lag:
            self.prev = rho[:7].clone()

    def distributions(self):
        return self.f.transpose(0, 1)


def exact(case, seed):
    if case["kind"] == "batch":
        out, left = [], 1500                       # steps that fit the time allowed
        for i, r in enumerate(_runs(case)):
            if r["steps"] > left:
                out.append(None)
                continue
            left -= r["steps"]
            small = r["shape"][0] * r["shape"][1] <= 3000
            e = _Exact(r["vset"], r["shape"], r["tau"], 1, "cpu" if small else "cuda", case["deriv"])
            e.init(_fields(r["shape"], r["amplitude"], r["direction"], 0.001, seed + 7919 * i).to(e.dev))
            for _ in range(r["steps"]):
                e.step()
            out.append(e.distributions().contiguous())
        return out
    shape, ad = _shape(case), case["kind"] == "ad"
    cells = shape[0] * shape[1] * shape[2]
    if cells * Q_OF[case["vset"]] * (2.3 if ad else 1) * case["steps"] > 6e9:
        return None
    e = _Exact(case["vset"], shape, case["tau"], SLICING[case["slicing"]],
               "cpu" if cells <= 3500 else "cuda", case.get("deriv", "sync"),
               case.get("shift", "none"), ad)
    e.init(_fields(shape, case["amplitude"], case["direction"], case["mix"], seed).to(e.dev))
    if ad:
        for _ in range(case["steps"]):
            e.step()
        return e.moments()
    got = []
    for _ in range(case["checks"]):
        for _ in range(case["steps"] // case["checks"]):
            e.step()
        got.append(e.moments())
    got = torch.stack(got)
    return [got, None] if case["monitor"] else got
