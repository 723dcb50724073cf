"""The runs whose speed counts, through the package's public calls.

A case is a dict of plain values with a "kind":
  run      start a lattice from a given state, advance it, read the state,
           the stress and the displacement back (what every user does)
  start    start and read-out alone, with the global diagnostics
  batch    many small specimens of uneven size advanced together
  adjoint  loss and gradients of a sensor misfit through torch.autograd

Edges are four letters (left, right, bottom, top): p periodic, v velocity
(clamped), t traction; "load" is the nominal traction of the right edge
(sin^2 ramp over 10000 steps), the other traction edges are free.

exact() restates the scheme (Feng & Chu, Sec. 3) in plain torch float64.
"""
import math
import random

import numpy as np
import torch

from paper_2605_26677_gb300 import lbm
from paper_2605_26677_gb300.autograd import SensorMisfit

LAWS = {"svk": lbm.LBM_LAW_SVK, "nh": lbm.LBM_LAW_NH, "lognh": lbm.LBM_LAW_LOGNH, "mr": lbm.LBM_LAW_MR,
        "yeoh": lbm.LBM_LAW_YEOH, "gent": lbm.LBM_LAW_GENT}
STORES = {"f64": lbm.LBM_STORE_F64, "f32": lbm.LBM_STORE_F32, "bf16": lbm.LBM_STORE_BF16, "f16": lbm.LBM_STORE_F16}
BCS = {"p": lbm.LBM_BC_PERIODIC, "v": lbm.LBM_BC_VELOCITY, "t": lbm.LBM_BC_TRACTION}
MODES, KMAX, AMP = 16, 8, 0.05   # the initial velocity field's Fourier modes
RAMP_STEPS = 10000
SENSORS, RECORD_EVERY = 64, 20
FLOPS_STEP, FLOPS_ADJOINT = 160, 400  # per node and step: collide-stream, its transpose


def _run(name, nx, ny, storage, edges, law, steps, omega=1.95, load=0.0, by=0.0):
    return {"name": name, "kind": "run", "nx": nx, "ny": ny, "storage": storage, "edges": edges, "law": law,
            "steps": steps, "omega": omega, "load": load, "by": by}


def listed():
    return [
        # the parity workload of the method: a 64^2 shear wave over 1000 steps; every step is launch and latency
        _run("shear_64_f64", 64, 64, "f64", "pppp", "nh", 1000, omega=2.0),
        # a test coupon of odd size with every edge rule: quick studies, parameter sweeps
        _run("coupon_131x37_f32", 131, 37, "f32", "vttt", "svk", 300, load=0.05),
        # the loaded specimen at 1/16 scale: what is run while a set-up is being found
        _run("specimen_256x128_f32", 256, 128, "f32", "vttt", "nh", 1250, load=0.3, by=-1e-6),
        # a strip, periodic along x, of ragged width: mid size, fits the L2 cache
        _run("strip_1000x517_f32", 1000, 517, "f32", "ppvt", "lognh", 301),
        # the loaded specimen at full size, in the default storage
        _run("specimen_4096x2048_f32", 4096, 2048, "f32", "vttt", "nh", 101, load=0.3, by=-1e-6),
        # the headline: waves in a periodic square of 67 M nodes
        _run("periodic_8192_f32", 8192, 8192, "f32", "pppp", "nh", 50, omega=2.0),
        # reduced-precision storage on both kinds of lattice
        _run("specimen_4096x2048_bf16", 4096, 2048, "bf16", "vttt", "nh", 101, load=0.3, by=-1e-6),
        _run("periodic_4096_f16", 4096, 4096, "f16", "pppp", "nh", 100, omega=2.0),
        # full precision at full size
        _run("specimen_4096x2048_f64", 4096, 2048, "f64", "vttt", "nh", 40, load=0.3, by=-1e-6),
        # a parameter study: 256 specimens of 64^2 to 1024^2 nodes, each with its own material and edges
        {"name": "batch_256_f32", "kind": "batch", "members": 256, "pick": 2, "storage": "f32", "steps": 40,
         "side_max": 1024},
        # one evaluation of an inverse problem: misfit at 64 sensors, gradients for mu(X) and v0
        {"name": "adjoint_1024_f32", "kind": "adjoint", "n": 1024, "storage": "f32", "steps": 200},
        # start from a strained state and read-out at full size (short runs, restarts, frequent output)
        {"name": "start_4096x2048_f32", "kind": "start", "nx": 4096, "ny": 2048, "storage": "f32", "edges": "vttt",
         "law": "nh", "omega": 1.95},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["run", "start", "batch", "adjoint"], [8, 1, 1, 1])[0]
    edges = rng.choice(["pppp", "pppp", "vttt", "vttt", "ppvt", "ppvv", "vvpp", "tvpp", "vvvv", "vvtt"])
    law = rng.choice(["nh", "nh", "nh", "svk", "lognh", "lognh", "mr", "yeoh", "gent"])
    if kind == "batch":
        return {"kind": "batch", "members": _log_int(rng, 8, 160), "pick": rng.randrange(1, 1000),
                "storage": rng.choice(["f32", "f32", "f64", "bf16", "f16"]), "steps": rng.randrange(9, 33),
                "side_max": _log_int(rng, 96, 700)}
    if kind == "adjoint":
        return {"kind": "adjoint", "n": _log_int(rng, 48, 700), "storage": rng.choice(["f32", "f32", "f64"]),
                "steps": RECORD_EVERY * rng.randrange(2, 8)}
    nx, ny = _log_int(rng, 24, 8192), _log_int(rng, 24, 8192)
    storage = rng.choice(["f32", "f32", "f32", "f64", "bf16", "f16"])
    while nx * ny > (12 << 20):
        nx, ny = (nx // 2 + rng.randrange(9), ny) if nx > ny else (nx, ny // 2 + rng.randrange(9))
    if kind == "start":
        return {"kind": "start", "nx": nx, "ny": ny, "storage": storage, "edges": edges, "law": "nh", "omega": 1.95}
    most = int(min(600, max(16, (160 << 20) / (nx * ny))))
    steps = rng.randrange(max(8, most // 2), most + 1)
    c = _run("", nx, ny, storage, edges, law, steps, omega=2.0 if edges == "pppp" else 1.95,
             load=0.2 if edges == "vttt" else 0.0, by=rng.choice([0.0, -1e-6]))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _params(law):
    """Closure parameters with lambda = 1.5, small-strain shear modulus 0.75."""
    return {"mr": [1.5, 0.25, 0.125], "yeoh": [1.5, 0.375, 0.05, 0.01], "gent": [1.5, 0.75, 20.0]}.get(law, [1.5, 0.75])


def _speed(lam, mu):
    return max(5.0, 3.0 * math.sqrt(lam + 2.0 * mu))


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _state(nx, ny, edges, seed):
    """U0 (6, ny, nx): F = I and a 16-mode velocity field of amplitude 0.05,
    windowed to zero at non-periodic edges."""
    dev, r = _device(), random.Random(seed)
    x = (torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) / nx
    y = (torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) / ny
    ay = torch.zeros((2, ny, 2 * MODES), dtype=torch.float64, device=dev)
    bx = torch.zeros((2 * MODES, nx), dtype=torch.float64, device=dev)
    for m in range(MODES):
        kx, ky = r.randint(-KMAX, KMAX) or 1, r.randint(-KMAX, KMAX)
        th, phi = 2 * math.pi * r.random(), 2 * math.pi * r.random()
        bx[2 * m], bx[2 * m + 1] = torch.cos(2 * math.pi * kx * x + phi), torch.sin(2 * math.pi * kx * x + phi)
        for k, w in ((0, math.cos(th)), (1, math.sin(th))):
            ay[k, :, 2 * m] = AMP / MODES * w * torch.cos(2 * math.pi * ky * y)
            ay[k, :, 2 * m + 1] = -AMP / MODES * w * torch.sin(2 * math.pi * ky * y)
    if edges[0] != "p":
        bx *= torch.sin(math.pi * x)
    if edges[2] != "p":
        ay *= torch.sin(math.pi * y)[None, :, None]
    U0 = torch.zeros((6, ny, nx), dtype=torch.float64, device=dev)
    U0[2] = U0[5] = 1.0
    U0[0], U0[1] = ay[0] @ bx, ay[1] @ bx
    return U0


def _fields(case, seed):
    """U0 and u0 of a run (from F = I and u = 0) or of a restart in a strained state ("start")."""
    U0 = _state(case["nx"], case["ny"], case["edges"], seed)
    if case["kind"] == "run":
        return U0, None
    for k in (1, 2):
        U0[2 * k:2 * k + 2] += _state(case["nx"], case["ny"], case["edges"], seed + 1000 * k)[:2]
    return U0, _state(case["nx"], case["ny"], case["edges"], seed + 3000)[:2].contiguous()


def _members(case, seed):
    """Sizes and edges by case["pick"]; materials by the seed: (nx, ny, edges, lam, mu)."""
    size, mat = random.Random(case["pick"]), random.Random(seed)
    out = []
    for _ in range(case["members"]):
        n = math.exp(2.0 * size.uniform(math.log(64 if case["side_max"] > 64 else 32), math.log(case["side_max"])))
        aspect = size.uniform(1.0, 4.0)
        nx, ny = max(3, round(math.sqrt(n * aspect))), max(3, round(math.sqrt(n / aspect)))
        edges = "v" + "".join(size.choice("vt") for _ in range(3))
        mu = mat.uniform(0.2, 2.0)
        out.append((nx, ny, edges, mu * mat.uniform(1.0, 4.0), mu))
    return out


def _inverse(case, seed):
    """mu = exp(0.3 g), g a Gaussian random field of correlation length n/16;
    a velocity pulse; sensors on the right edge; target readings."""
    n, dev = case["n"], _device()
    r = np.random.RandomState(seed % (1 << 32))
    k = 2 * math.pi * np.fft.fftfreq(n)
    g = np.fft.ifft2(np.fft.fft2(r.standard_normal((n, n))) *
                     np.exp(-(k[:, None] ** 2 + k[None, :] ** 2) * (n / 16.0) ** 2 / 4)).real
    mu = np.exp(0.3 * (g - g.mean()) / g.std())
    th = 2 * math.pi * r.rand()
    X = np.arange(n) + 0.5
    pulse = 0.01 * np.exp(-((X[None, :] - 0.9 * n) ** 2 + (X[:, None] - 0.5 * n) ** 2) / (2 * (n / 16.0) ** 2))
    v0 = np.stack([math.cos(th) * pulse, math.sin(th) * pulse])
    ns = min(SENSORS, n // 2)
    sens = np.array([[n - 1, int((j + 0.5) * n / ns)] for j in range(ns)], dtype=np.int32)
    rec = np.arange(RECORD_EVERY, case["steps"] + 1, RECORD_EVERY, dtype=np.int32)
    target = 1e-3 * (2 * r.rand(len(rec), ns, 2) - 1)
    return {"mu": torch.from_numpy(mu).to(dev), "v0": torch.from_numpy(v0).to(dev), "sensors": sens, "records": rec,
            "target": target, "c": max(5.0, 3.0 * math.sqrt(4.0 * mu.max())), "omega": 1.95}


# ---------------------------------------------------------------- the library's side
def _lattice(nx, ny, storage, edges, law, params, c, omega, load=0.0, by=0.0):
    L = lbm.Lattice(nx, ny, dx=1.0, c=c, omega=omega, storage=STORES[storage])
    lbm.lbm_set_material(L.ctx, LAWS[law], params)
    lbm.lbm_set_body_force(L.ctx, 0.0, by)
    for e, kind in enumerate(edges):
        if kind != "p":
            tf = lbm.LBM_T_SIN2_RAMP if e == 1 and load else lbm.LBM_T_CONST
            lbm.lbm_set_boundary(L.ctx, e, BCS[kind], (load if e == 1 else 0.0, 0.0), tf, (RAMP_STEPS / c, 0, 0, 0))
    return L


class _Run:
    """One lattice with its start state and the arrays that the results are read into."""

    def __init__(self, case, seed):
        nx, ny = case["nx"], case["ny"]
        p = _params(case["law"])
        self.L = _lattice(nx, ny, case["storage"], case["edges"], case["law"], p, _speed(1.5, 0.75), case["omega"],
                          case.get("load", 0.0), case.get("by", 0.0))
        self.steps = case.get("steps", 0)
        self.diag = case["kind"] == "start"
        self.U0, self.u0 = _fields(case, seed)
        self.U, self.P, self.u = (torch.empty((k, ny, nx), dtype=torch.float64, device=_device()) for k in (6, 4, 2))

    def __call__(self):
        ctx = self.L.ctx
        lbm.lbm_init_device(ctx, self.U0, self.u0)
        if self.steps:
            lbm.lbm_step(ctx, self.steps)
        lbm.lbm_read_state_device(ctx, self.U, self.P)
        lbm.lbm_read_displacement_device(ctx, self.u)
        out = [self.U, self.P, self.u]
        return out + [lbm.lbm_diagnostics(ctx)] if self.diag else out


class _Batch:
    """Specimens advanced together, their results in two flat arrays."""

    def __init__(self, case, seed):
        mem = _members(case, seed)
        self.steps = case["steps"]
        self.lat = [_lattice(nx, ny, case["storage"], ed, "nh", [lam, mu], _speed(lam, mu), 1.95)
                    for nx, ny, ed, lam, mu in mem]
        self.U0 = [_state(nx, ny, ed, seed + k) for k, (nx, ny, ed, _, _) in enumerate(mem)]
        total = sum(m[0] * m[1] for m in mem)
        self.U, self.u = (torch.empty(k * total, dtype=torch.float64, device=_device()) for k in (6, 2))
        self.parts, at = [], 0
        for nx, ny, _, _, _ in mem:
            n = nx * ny
            self.parts.append((self.U[6 * at:6 * (at + n)], self.u[2 * at:2 * (at + n)]))
            at += n
        for L, U0 in zip(self.lat, self.U0):
            lbm.lbm_init_device(L.ctx, U0)
        self.batch = lbm.lbm_batch_create([L.ctx for L in self.lat])
        lbm.lbm_batch_tune(self.batch, 4)

    def __call__(self):
        for L, U0 in zip(self.lat, self.U0):
            lbm.lbm_init_device(L.ctx, U0)
        lbm.lbm_batch_step(self.batch, self.steps, graph_steps=8)
        for L, (U, u) in zip(self.lat, self.parts):
            lbm.lbm_read_state_device(L.ctx, U)
            lbm.lbm_read_displacement_device(L.ctx, u)
        return [self.U, self.u]

    def __del__(self):
        lbm.lbm_batch_destroy(getattr(self, "batch", None))


class _Adjoint:
    """A misfit with its checkpoints, and the fields that it is differentiated by."""

    def __init__(self, case, seed):
        w = _inverse(case, seed)
        n = case["n"]
        self.mu, self.v0 = w["mu"].requires_grad_(), w["v0"].requires_grad_()
        self.misfit = SensorMisfit(n, n, w["c"], w["omega"], [("velocity", (0.0, 0.0))] + 3 * [("traction", (0.0, 0.0))],
                                   w["sensors"], w["records"], w["target"], case["steps"],
                                   storage=STORES[case["storage"]])

    def __call__(self):
        loss = self.misfit(self.mu, self.v0)
        gmu, gv0 = torch.autograd.grad(loss, (self.mu, self.v0))
        return [loss.detach(), gmu, gv0]

    def __del__(self):
        if hasattr(self, "misfit"):
            self.misfit.close()


def prepare(case, seed):
    return {"run": _Run, "start": _Run, "batch": _Batch, "adjoint": _Adjoint}[case["kind"]](case, seed)


def run(state):
    return state()


def work(case):
    """Start state in, results out, each once; the arithmetic of every step."""
    if case["kind"] == "adjoint":
        n = case["n"] ** 2
        return {"bytes": n * 8 * (3 + 3), "flops": n * case["steps"] * (FLOPS_STEP + FLOPS_ADJOINT)}
    if case["kind"] == "batch":
        n = sum(m[0] * m[1] for m in _members(case, 0))
        return {"bytes": n * 8 * (6 + 8), "flops": n * case["steps"] * FLOPS_STEP}
    n = case["nx"] * case["ny"]
    return {"bytes": n * 8 * (6 + 12), "flops": n * (case.get("steps", 0) + 2) * FLOPS_STEP}


# ---------------------------------------------------------------- 64-bit restatement
CI, CJ = (1, 0, -1, 0), (0, 1, 0, -1)          # Sec. 3.1
DMISS, DOUT = (0, 2, 1, 3), (2, 0, 3, 1)       # missing and outgoing direction per edge


def _piola(law, p, F):
    """P = dW/dF (Appendix A) of F = (F11, F12, F21, F22), real or complex."""
    J = F[0] * F[3] - F[1] * F[2]
    H = [F[3] / J, -F[2] / J, -F[1] / J, F[0] / J]
    lam, mu = p[0], p[1]
    if law == "svk":
        E11 = 0.5 * (F[0] * F[0] + F[2] * F[2] - 1.0)
        E22 = 0.5 * (F[1] * F[1] + F[3] * F[3] - 1.0)
        S12 = mu * (F[0] * F[1] + F[2] * F[3])
        S11, S22 = lam * (E11 + E22) + 2 * mu * E11, lam * (E11 + E22) + 2 * mu * E22
        return [F[0] * S11 + F[1] * S12, F[0] * S12 + F[1] * S22, F[2] * S11 + F[3] * S12, F[2] * S12 + F[3] * S22]
    if law in ("nh", "lognh"):
        a = 0.5 * lam * (J * J - 1.0) if law == "nh" else lam * torch.log(J)
        return [mu * (F[m] - H[m]) + a * H[m] for m in range(4)]
    tr = F[0] * F[0] + F[1] * F[1] + F[2] * F[2] + F[3] * F[3]
    lJ = torch.log(J)
    I1, I2, j23, j43 = tr + 1.0, J * J + tr, torch.exp(-2.0 / 3.0 * lJ), torch.exp(-4.0 / 3.0 * lJ)
    A = j23 * I1 - 3.0
    s1 = p[1] if law == "mr" else p[1] + 2 * p[2] * A + 3 * p[3] * A * A if law == "yeoh" else p[1] / (2 * (1 - A / p[2]))
    P = [s1 * j23 * (2 * F[m] - 2.0 / 3.0 * I1 * H[m]) + lam * lJ * H[m] for m in range(4)]
    if law == "mr":
        P = [P[m] + p[2] * j43 * (2 * F[m] + (2 * J * J - 4.0 / 3.0 * I2) * H[m]) for m in range(4)]
    return P


def _jvp(law, p, F, dF):
    """C : dF by the complex step."""
    h = 1e-30
    return [Pm.imag / h for Pm in _piola(law, p, [torch.complex(f, h * d) for f, d in zip(F, dF)])]


def _diff(a, dim, periodic):
    """Second-order difference of Sec. 3.4 at dx = 1."""
    d = 0.5 * (torch.roll(a, -1, dim) - torch.roll(a, 1, dim))
    if not periodic:
        s = [a.select(dim, i) for i in (0, 1, 2, -1, -2, -3)]
        d.select(dim, 0).copy_(0.5 * (-3 * s[0] + 4 * s[1] - s[2]))
        d.select(dim, -1).copy_(0.5 * (3 * s[3] - 4 * s[4] + s[5]))
    return d


class _Exact:
    """The scheme on one lattice; p[1] may be a field (with p[0] = ratio * p[1])."""

    def __init__(self, nx, ny, edges, law, p, c, omega, load=0.0, by=0.0):
        self.nx, self.ny, self.edges, self.law, self.p, self.c, self.w = nx, ny, edges, law, p, c, omega
        self.dt, self.load, self.by, self.n = 1.0 / c, load, by, 0

    def _flux(self, U, P):
        return [-P[0], -P[2], -U[0], None, -U[1], None], [-P[1], -P[3], None, -U[0], None, -U[1]]

    def _feq(self, U, P):
        out = []
        for q in range(4):
            phi, s = self._flux(U, P)[q & 1], (1.0, 1.0, -1.0, -1.0)[q]
            out.append([0.25 * U[k] if phi[k] is None else 0.25 * U[k] + (0.5 * s / self.c) * phi[k] for k in range(6)])
        return out

    def start(self, U0, u0=None):
        """Eqs. (16)-(21) and u*^0 = u0 - (dt/2) v0."""
        px, py, c, b = self.edges[0] == "p", self.edges[2] == "p", self.c, (0.0, self.by)
        U = [U0[k] for k in range(6)]
        f = self._feq(U, _piola(self.law, self.p, U[2:]))
        gX, gY = [_diff(a, 1, px) for a in U], [_diff(a, 0, py) for a in U]
        tan = self.tangent if hasattr(self, "tangent") else lambda d: _jvp(self.law, self.p, U[2:], d)
        dX, dY = tan(gX[2:]), tan(gY[2:])
        rate = [b[0] + dX[0] + dY[1], b[1] + dX[2] + dY[3], gX[0], gY[0], gX[1], gY[1]]
        for q in range(4):
            i, j = CI[q], CJ[q]
            Z = [rate[k] + c * i * gX[k] + c * j * gY[k] for k in range(6)]
            dP = tan(Z[2:])
            D = [Z[0] - 2 / c * (i * dP[0] + j * dP[1]), Z[1] - 2 / c * (i * dP[2] + j * dP[3]),
                 Z[2] - 2 * i / c * Z[0], Z[3] - 2 * j / c * Z[0], Z[4] - 2 * i / c * Z[1], Z[5] - 2 * j / c * Z[1]]
            f[q] = torch.stack([f[q][k] - 0.125 * self.dt * D[k] for k in range(6)])
        self.f, self.ustar, self.n = f, -0.5 * self.dt * U0[:2] + (0.0 if u0 is None else u0), 0

    def state(self):
        U = list(self.f[0] + self.f[1] + self.f[2] + self.f[3])
        U[1] = U[1] + 0.5 * self.dt * self.by
        return U

    def _at(self, e, a):
        return a[..., 0] if e == 0 else a[..., -1] if e == 1 else a[..., 0, :] if e == 2 else a[..., -1, :]

    def _traction(self, U, T):
        """F^b of every traction edge at once (Sec. 3.6.2, node form)."""
        es = [e for e in range(4) if self.edges[e] == "t"]
        lens = [self.ny if e < 2 else self.nx for e in es]
        isx = torch.cat([torch.full((n,), e < 2, device=U[0].device) for e, n in zip(es, lens)])
        sgn = torch.cat([torch.full((n,), -1.0 if e in (0, 2) else 1.0, dtype=torch.float64, device=U[0].device)
                         for e, n in zip(es, lens)])
        F = [torch.cat([self._at(e, U[2 + m]) for e in es]) for m in range(4)]
        p = [torch.cat([self._at(e, v) for e in es]) if torch.is_tensor(v) else v for v in self.p]
        Tb = [torch.cat([torch.full((n,), T[e][i], dtype=torch.float64, device=U[0].device)
                         for e, n in zip(es, lens)]) for i in range(2)]
        tang = [torch.where(isx, F[2 * i + 1], F[2 * i]) for i in range(2)]
        norm = [torch.where(isx, F[2 * i], F[2 * i + 1]) for i in range(2)]

        def full(nv, tv):
            return [torch.where(isx, nv[0], tv[0]), torch.where(isx, tv[0], nv[0]),
                    torch.where(isx, nv[1], tv[1]), torch.where(isx, tv[1], nv[1])]

        def residual(P):
            return [sgn * torch.where(isx, P[2 * i], P[2 * i + 1]) - Tb[i] for i in range(2)]

        def jac(nv, tv):
            h, one, zero = 1e-30, torch.ones_like(sgn), torch.zeros_like(sgn)
            cols = []
            for d in ((one, zero), (zero, one)):
                P = _piola(self.law, [v.detach() if torch.is_tensor(v) else v for v in p],
                           full([torch.complex(nv[i], h * d[i]) for i in range(2)],
                                [torch.complex(tv[i], zero) for i in range(2)]))
                r = [sgn * torch.where(isx, P[2 * i], P[2 * i + 1]) for i in range(2)]
                cols.append([x.imag / h for x in r])
                res = [r[i].real - Tb[i] for i in range(2)]
            return res, cols

        def solve(r, cols):
            det = cols[0][0] * cols[1][1] - cols[1][0] * cols[0][1]
            return [(cols[1][1] * r[0] - cols[1][0] * r[1]) / det, (cols[0][0] * r[1] - cols[0][1] * r[0]) / det]

        with torch.no_grad():
            nv, tv = [x.detach().clone() for x in norm], [x.detach() for x in tang]
            for _ in range(12):
                r, cols = jac(nv, tv)
                nv = [a - d for a, d in zip(nv, solve(r, cols))]
                if max(float(x.abs().max()) for x in r) < 1e-9:  # the step just made squares it
                    break
            cols = jac(nv, tv)[1]
        if any(x.requires_grad for x in tang) or any(torch.is_tensor(v) and v.requires_grad for v in p):
            # one more Newton step carries the derivative of the solution
            nv = [a - d for a, d in zip(nv, solve(residual(_piola(self.law, p, full(nv, tang))), cols))]
        Fb = full(nv, tang)
        out, at = {}, 0
        for e, n in zip(es, lens):
            out[e] = [x[at:at + n] for x in Fb]
            at += n
        return out

    def step(self):
        """One step of Sec. 3.7."""
        c, w, dt = self.c, self.w, self.dt
        U = self.state()
        self.ustar = self.ustar + dt * torch.stack(U[:2])
        P = _piola(self.law, self.p, U[2:])
        phis, src = self._flux(U, P), dt * (2 - w) * 0.125 * self.by
        fs = []
        for q in range(4):
            s = (0.5 * w / c) * (1.0, 1.0, -1.0, -1.0)[q]
            col = []
            for k in range(6):
                a = (1 - w) * self.f[q][k] + (0.25 * w) * U[k]
                if phis[q & 1][k] is not None:
                    a = a + s * phis[q & 1][k]
                col.append(a + src if k == 1 else a)
            fs.append(torch.stack(col))
            if not torch.is_grad_enabled():
                self.f[q] = None
        th = (self.n + 0.5) * dt
        g = math.sin(math.pi * th / (2 * RAMP_STEPS * dt)) ** 2 if th < RAMP_STEPS * dt else 1.0
        T = [(self.load * g if e == 1 else 0.0, 0.0) for e in range(4)]
        Fb = self._traction(U, T) if "t" in self.edges else {}
        new = [torch.roll(fs[q], (CI[q] or CJ[q]), 2 if CI[q] else 1) for q in range(4)]
        for e, kind in enumerate(self.edges):
            if kind == "p":
                continue
            d, out = DMISS[e], self._at(e, fs[DOUT[e]])
            if kind == "v":   # Eq. (24) with v_D = 0
                val = torch.cat([-out[:2], out[2:]])
            else:             # Eq. (25); F^b / 2 and D = -1 on the F-components
                val = torch.cat([torch.stack([out[i] + T[e][i] / c for i in range(2)]),
                                 0.5 * torch.stack(Fb[e]) - out[2:]])
            self._at(e, new[d]).copy_(val)
        self.f, self.n = new, self.n + 1

    def results(self):
        U = self.state()
        return [torch.stack(U), torch.stack(_piola(self.law, self.p, U[2:])),
                self.ustar + 0.5 * self.dt * torch.stack(U[:2])]


def _exact_run(case, seed):
    X = _Exact(case["nx"], case["ny"], case["edges"], case["law"], _params(case["law"]), _speed(1.5, 0.75),
               case["omega"], case.get("load", 0.0), case.get("by", 0.0))
    X.start(*_fields(case, seed))
    for _ in range(case.get("steps", 0)):
        X.step()
    out = X.results()
    if case["kind"] == "run":
        return out
    U, (lam, mu) = out[0], _params("nh")
    F = U[2:]
    J = F[0] * F[3] - F[1] * F[2]
    W = 0.5 * mu * ((F * F).sum(0) - 2 - 2 * torch.log(J)) + 0.25 * lam * (J * J - 1 - 2 * torch.log(J))
    G = F - torch.tensor([1.0, 0, 0, 1.0], dtype=torch.float64, device=F.device)[:, None, None]
    d = [U[0].sum(), U[1].sum()] + [F[m].mean() for m in range(4)]
    d += [(0.5 * (U[0] ** 2 + U[1] ** 2) + W).sum(), J.min(), J.max(), (G * G).sum(0).sqrt().max()]
    return out + [torch.stack(d)]


def _exact_batch(case, seed):
    U, u = [], []
    for k, (nx, ny, ed, lam, mu) in enumerate(_members(case, seed)):
        X = _Exact(nx, ny, ed, "nh", [lam, mu], _speed(lam, mu), 1.95)
        X.start(_state(nx, ny, ed, seed + k))
        for _ in range(case["steps"]):
            X.step()
        r = X.results()
        U.append(r[0].reshape(-1))
        u.append(r[2].reshape(-1))
    return [torch.cat(U), torch.cat(u)]


def _exact_adjoint(case, seed):
    from torch.utils.checkpoint import checkpoint

    w, n = _inverse(case, seed), case["n"]
    mu, v0 = w["mu"].requires_grad_(), w["v0"].requires_grad_()
    target = torch.from_numpy(w["target"]).to(mu.device)
    sx, sy = (torch.from_numpy(w["sensors"][:, i].astype(np.int64)).to(mu.device) for i in (0, 1))

    def lattice(m):
        X = _Exact(n, n, "vttt", "nh", [2.0 * m, m], w["c"], w["omega"])
        # the start's tangent at F = I
        X.tangent = lambda d: [2 * m * (d[0] + d[3]) + 2 * m * d[0], m * (d[1] + d[2]), m * (d[1] + d[2]),
                               2 * m * (d[0] + d[3]) + 2 * m * d[3]]
        return X

    def segment(m, f, ustar, at):
        X = lattice(m)
        X.f, X.ustar, X.n = list(f), ustar, at
        for _ in range(RECORD_EVERY):
            X.step()
        r = (X.ustar + 0.5 * X.dt * torch.stack(X.state()[:2]))[:, sy, sx].T - target[at // RECORD_EVERY]
        return torch.stack(X.f), X.ustar, 0.5 * (r * r).sum()

    X = lattice(mu)
    X.start(torch.cat([v0, torch.ones_like(v0[:1]), torch.zeros_like(v0), torch.ones_like(v0[:1])]))
    f, ustar, loss = torch.stack(X.f), X.ustar, 0.0
    for at in range(0, case["steps"], RECORD_EVERY):
        f, ustar, part = checkpoint(segment, mu, f, ustar, at, use_reentrant=False)
        loss = loss + part
    g = torch.autograd.grad(loss, (mu, v0))
    return [loss.detach(), g[0], g[1]]


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    with torch.no_grad():
        return _exact_batch(case, seed) if case["kind"] == "batch" else _exact_run(case, seed)
