"""The calls a program makes of this library, as timing cases.

A case is one call (or one short sequence of calls) through the public Python
binding of the C ABI on fields that live on the GPU:

  forward     march a velocity field a few time steps (a direct simulation)
  adjoint     one adjoint step about a stored state (a caller's own sweep)
  gradient    the checkpointed gradient of the final energy, the unit of work
              of the optimal-perturbation search
  continuous  the same gradient through the continuous adjoint equations
  batch       several gradient requests with their own physics in one batch
              (the serving form)

Grids, physics and precisions are those of the benchmark, the tests and the
paper's runs; `draw` spreads over the same ranges, odd radial sizes and
transform lengths without a register FFT among them.

`exact` is a plain torch FP64 restatement of the discrete scheme (dense radial
matrices, library FFTs, the adjoint by automatic differentiation of the step).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_10103_gb300 import _lib as pnop

PRECISION = {"fp64": pnop.PNOP_FP64, "mixed": pnop.PNOP_MIXED, "df": pnop.PNOP_DF, "mixed_df": pnop.PNOP_MIXED_DF}


def _case(name, kind, grid, precision, steps, snaps=1, count=1, Lz=10.0, Re=2000.0, dt=0.005, Wo=8.0, A=1.0, E0=1e-6,
          decay=4.0):
    nr, ntheta, nz = grid
    c = dict(kind=kind, nr=nr, ntheta=ntheta, nz=nz, precision=precision, steps=steps, snaps=snaps, count=count, Lz=Lz,
             Re=Re, dt=dt, Wo=Wo, A=A, E0=E0, decay=decay)
    return dict(c, name=name) if name else c


BIG = dict(Lz=100.0, Re=2000.0, dt=0.0025, decay=12.0)  # the benchmark's physics
CFG2 = dict(Lz=50.0, Re=2500.0, dt=0.005, decay=8.0)    # the FP64-against-mixed workload


def listed():
    return [
        # one time step on the smallest serving resolution: the smallest call, launches and latency
        _case("step_32x32x64_mixed_df", "forward", (32, 32, 64), "mixed_df", 1),
        # the plain FP64 gradient of the small configuration (100 of its 200 steps)
        _case("grad_32x16x32_fp64", "gradient", (32, 16, 32), "fp64", 100, snaps=8, dt=0.01),
        # 16 serving requests of the smallest resolution in one batch
        _case("batch16_32x32x64_mixed", "batch", (32, 32, 64), "mixed", 20, snaps=8, count=16),
        # 8 serving requests of the middle resolution in one batch
        _case("batch8_48x48x128_mixed", "batch", (48, 48, 128), "mixed", 10, snaps=8, count=8, Lz=50.0, decay=8.0),
        # the gradient of the precision comparison's grid, in both precisions (Stockham transform lengths)
        _case("grad_48x32x96_fp64", "gradient", (48, 32, 96), "fp64", 20, snaps=8, **CFG2),
        _case("grad_48x32x96_mixed", "gradient", (48, 32, 96), "mixed", 40, snaps=8, **CFG2),
        # the continuous adjoint, the form the paper integrates
        _case("cont_48x48x128_mixed_df", "continuous", (48, 48, 128), "mixed_df", 10, snaps=8, Lz=50.0, decay=8.0),
        # a radial grid above 64 points and lengths with more 3s than 2s
        _case("grad_81x36x108_mixed_df", "gradient", (81, 36, 108), "mixed_df", 10, snaps=6, Lz=25.0, decay=8.0),
        # the headline grid: marching, one adjoint step, the checkpointed gradient, and the FP64 gradient
        _case("march_64x64x256_mixed_df", "forward", (64, 64, 256), "mixed_df", 4, **BIG),
        _case("adj_64x64x256_mixed_df", "adjoint", (64, 64, 256), "mixed_df", 1, E0=1e-7, **BIG),
        _case("grad_64x64x256_mixed_df", "gradient", (64, 64, 256), "mixed_df", 20, snaps=12, **BIG),
        _case("grad_64x64x256_fp64", "gradient", (64, 64, 256), "fp64", 8, snaps=5, **BIG),
    ]


def draw(rng):
    limit = 64 * 64 * 256 * 20 * 3  # values times step-equivalents of the largest listed case
    while True:
        nr = int(round(math.exp(rng.uniform(math.log(16), math.log(96)))))
        ntheta = 2 * rng.choice([4, 6, 8, 9, 12, 16, 18, 24, 27, 32])
        nz = 2 * rng.choice([8, 12, 16, 18, 24, 27, 32, 36, 48, 54, 64, 72, 96, 128])
        kind = rng.choice(["forward", "adjoint", "gradient", "gradient", "continuous", "batch"])
        precision = rng.choice(["fp64", "mixed", "mixed", "df", "mixed_df", "mixed_df"])
        steps = {"forward": rng.randint(1, 6), "adjoint": 1}.get(kind, rng.randint(2, 30))
        snaps = rng.randint(2, 8) if kind in ("gradient", "continuous", "batch") else 1
        count = rng.randint(2, 16) if kind == "batch" else 1
        slow = 6 if precision in ("fp64", "df") else 1
        cost = nr * ntheta * nz * steps * count * slow * (1 if kind in ("forward", "adjoint") else 3)
        if cost > limit or nr * ntheta * nz * count > 8 * 64 * 64 * 256:
            continue
        return _case("", kind, (nr, ntheta, nz), precision, steps, snaps, count, Lz=rng.choice([10.0, 25.0, 50.0, 100.0]),
                     Re=round(rng.uniform(1500.0, 3000.0), 1), dt=rng.choice([0.0025, 0.005, 0.01]),
                     Wo=round(rng.uniform(4.0, 18.0), 2), A=round(rng.uniform(0.5, 1.5), 2),
                     E0=1e-7 if kind == "adjoint" else 10.0 ** round(rng.uniform(-7, -6), 1), decay=rng.choice([4.0, 8.0, 12.0]))


def _dims(case):
    M, K = case["ntheta"] // 2 - 1, case["nz"] // 2 - 1
    return case["nr"], M, K, 2 * M + 1, K + 1


def _requests(case, seed):
    """Physics and energy of every request: the case's own, or seeded ones around it for a batch."""
    out = []
    rng = np.random.default_rng(1000 + seed)
    for i in range(case["count"]):
        q = {k: case[k] for k in ("Re", "dt", "Wo", "A", "E0")}
        q["tau0"] = 0.25 * 2.0 * math.pi * case["Re"] / case["Wo"] ** 2  # start of the deceleration
        if case["kind"] == "batch":
            q.update(Re=float(rng.uniform(1500, 3000)), Wo=float(rng.uniform(4, 18)), A=float(rng.uniform(0.5, 1.5)),
                     E0=float(10.0 ** rng.uniform(-7, -6)), tau0=float(rng.uniform(0, 50)))
        out.append(q)
    return out


def _field(case, seed, amplitude=None):
    """A seeded solenoidal field, zero at the wall, every mode excited with amplitude
    exp(-sqrt(m^2 + k^2) / decay): u = curl(psi e_z) + curl curl(phi e_z) with
    psi = (1 - r^2)^2 r^|m| P(r^2), phi = (1 - r^2)^3 r^|m| Q(r^2)."""
    nr, M, K, nm, nk = _dims(case)
    gen = torch.Generator().manual_seed(int(seed))
    c = torch.randn(2, 2, 2, nm, nk, generator=gen, dtype=torch.float64)  # (P or Q, re or im, power, m, k)
    c = torch.complex(c[:, 0], c[:, 1])
    m = torch.arange(-M, M + 1, dtype=torch.float64)[:, None]
    k = torch.arange(nk, dtype=torch.float64)[None, :]
    c = c * torch.exp(-torch.sqrt(m * m + k * k) / case["decay"])
    c[:, :, :M, 0] = c[:, :, M + 1:, 0].flip(-1).conj()  # a real field: Hermitian k = 0 plane
    c[:, :, M, 0] = c[:, :, M, 0].real.to(c.dtype)
    dev = "cuda"
    c, m = c.to(dev), m.to(dev)
    kz = (2.0 * math.pi / case["Lz"]) * k.to(dev)
    j = torch.arange(nr, dtype=torch.float64, device=dev)
    r = torch.cos(math.pi * j / (2 * nr - 1))
    r[0] = 1.0
    am = m.abs()

    def power(p, shift):  # r^(|m| + p - shift), 0 where the exponent is negative (its factor is 0 there)
        e = am + p - shift
        return torch.where(e >= 0, r[:, None, None] ** e.clamp(min=0), torch.zeros((), device=dev, dtype=r.dtype))

    def poly(base, a):  # coefficients in r^2 of (1 - s)^base (a0 + a1 s)
        w = [1.0]
        for _ in range(base):
            w = [x - y for x, y in zip(w + [0.0], [0.0] + w)]
        return [(w[i] if i < len(w) else 0.0) * a[0] + (w[i - 1] if i else 0.0) * a[1] for i in range(base + 2)]

    u = torch.zeros(3, nr, nm, nk, dtype=torch.complex128, device=dev)
    for i, q in enumerate(poly(2, c[0])):
        n = am + 2 * i
        u[0] += 1j * m * q * power(2 * i, 1)
        u[1] -= n * q * power(2 * i, 1)
    for i, q in enumerate(poly(3, c[1])):
        n = am + 2 * i
        u[0] += 1j * kz * n * q * power(2 * i, 1)
        u[1] -= m * kz * q * power(2 * i, 1)
        u[2] -= (n * n - m * m) * q * power(2 * i, 2)
    u[:, 0] = 0.0
    u[:, :, M, 0] = u[:, :, M, 0].real.to(u.dtype)
    u[0, :, M, 0] = 0.0
    u[2, :, M, 0] = 0.0
    return u if amplitude is None else u * (amplitude / u.abs().max())


def _amplitude(case):
    """Largest coefficient of a state of energy about E0: its root mean square over the pipe."""
    return math.sqrt(2.0 * case["E0"] / (math.pi * case["Lz"]))


class _Ops:
    """The host operators of a batch's requests, freed with it."""

    def __init__(self, batch, requests):
        self.free = pnop.Batch.pnop_ops_free
        self.all = [batch.pnop_batch_prepare(q["Re"], q["dt"], q["Wo"], q["A"], q["tau0"]) for q in requests]

    def __del__(self):
        for o in self.all:
            self.free(o)


def prepare(case, seed):
    requests = _requests(case, seed)
    q = requests[0]
    prec = PRECISION[case["precision"]]
    s = {"case": case}
    grid = (case["nr"], case["ntheta"], case["nz"], case["Lz"])
    if case["kind"] == "batch":
        s["batch"] = pnop.Batch(*grid, capacity=case["count"], precision=prec, snap_budget=case["snaps"])
        s["requests"] = requests
        s["ops"] = _Ops(s["batch"], requests)
        s["u0"] = [_field(case, 100 * seed + i) for i in range(case["count"])]
        s["g"] = [torch.zeros_like(u) for u in s["u0"]]
        return s
    s["ctx"] = pnop.Context(*grid, q["Re"], q["dt"], q["Wo"], q["A"], q["tau0"], prec, case["snaps"])
    s["t"] = q["tau0"]
    s["u0"] = _field(case, 100 * seed, _amplitude(case) if case["kind"] in ("forward", "adjoint") else None)
    if case["kind"] == "adjoint":
        s["lam0"] = _field(case, 100 * seed + 50, 1.0)
    s["out"] = torch.zeros_like(s["u0"])
    return s


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        b = state["batch"]
        ids = [b.pnop_batch_submit_prepared(o, u, q["E0"], case["steps"] * q["dt"])
               for o, u, q in zip(state["ops"].all, state["u0"], state["requests"])]
        b.pnop_batch_run(1 << 30)
        gains = [b.pnop_batch_result(i, g) for i, g in zip(ids, state["g"])]
        return {"gradient": state["g"], "gain": np.array(gains)}
    ctx, out = state["ctx"], state["out"]
    if kind == "forward":
        out.copy_(state["u0"])
        ctx.pnop_step_forward(out, state["t"], case["steps"])
        return {"u": out}
    if kind == "adjoint":
        out.copy_(state["lam0"])
        ctx.pnop_step_adjoint(state["u0"], out, state["t"])
        return {"lam": out}
    call = ctx.pnop_gradient if kind == "gradient" else ctx.pnop_gradient_continuous
    gain = call(state["u0"], case["E0"], case["steps"] * case["dt"], out)
    return {"gradient": out, "gain": gain}


def work(case):
    """Each input field read and each output field written once; per time step two
    nonlinear terms (9 transforms in theta and z each, curl, products) and two stages
    (one pressure and three Helmholtz banded solves per mode, divergence, gradient,
    corrections); an adjoint step re-runs the predictor and transposes both stages
    and both nonlinear terms (6 + 9 transforms)."""
    nr, M, K, nm, nk = _dims(case)
    nt, nz, S = 3 * (M + 1), 3 * (K + 1), nr * nm * nk
    fft = 5.0 * nr * nk * nt * math.log2(nt) + 2.5 * nr * nt * nz * math.log2(nz)  # one field
    curl, stage = 100.0 * S, (4 * 2 * 2 * 9 + 150.0) * S
    fwd = 2 * (9 * fft + 9.0 * nr * nt * nz + curl + stage)
    adj = (9 + 15 + 9) * fft + 45.0 * nr * nt * nz + 4 * curl + 3.5 * stage
    cont = 2 * (21 * fft + 45.0 * nr * nt * nz + 2.5 * curl + stage)
    n, kind = case["steps"], case["kind"]
    flops = {"forward": n * fwd, "adjoint": adj, "continuous": n * (fwd + cont)}.get(kind, n * (fwd + adj))
    fields = 3 if kind == "adjoint" else 2
    return {"bytes": case["count"] * fields * 48.0 * S, "flops": case["count"] * flops}


# ---------------------------------------------------------------- plain torch FP64 restatement
def _fd(x0, x):
    """Weights of the first and second derivative at x0 on the nodes x (Vandermonde, extended precision)."""
    x = np.asarray(x, np.longdouble) - np.longdouble(x0)
    h = np.abs(x).max()
    n = len(x)
    A = np.array([(x / h) ** p for p in range(n)], np.longdouble)
    B = np.zeros((n, 2), np.longdouble)
    B[1, 0], B[2, 1] = 1.0 / h, 2.0 / h ** 2
    for c in range(n):  # Gauss elimination with partial pivoting in extended precision
        p = c + int(np.argmax(np.abs(A[c:, c])))
        A[[c, p]], B[[c, p]] = A[[p, c]], B[[p, c]]
        f = A[c + 1:, c] / A[c, c]
        A[c + 1:] -= f[:, None] * A[c]
        B[c + 1:] -= f[:, None] * B[c]
    for c in range(n - 1, -1, -1):
        B[c] = (B[c] - A[c, c + 1:] @ B[c + 1:]) / A[c, c]
    return B.astype(np.float64)


def _bessel(nu, z):
    term = (z / 2.0) ** nu / math.factorial(nu)
    total = term
    for k in range(1, 200):
        term = term * (-(z / 2.0) ** 2) / (k * (k + nu))
        total = total + term
    return total


class _Plain:
    """The discrete scheme with dense radial matrices, batched over the modes."""

    def __init__(self, case, q):
        self.q, self.case = q, case
        nr, M, K, nm, nk = self.dims = _dims(case)
        self.nt, self.nz = 3 * (M + 1), 3 * (K + 1)
        dev = dict(device="cuda", dtype=torch.float64)
        r = np.cos(np.pi * np.arange(nr) / (2 * nr - 1))
        ext = np.r_[r, -r[::-1]]
        D1, D2 = np.zeros((2, nr, nr)), np.zeros((2, nr, nr))  # even, odd parity at the axis
        for j in range(nr):
            lo = min(max(j - 4, 0), 2 * nr - 9)
            w = _fd(r[j], ext[lo:lo + 9])
            for t, e in enumerate(range(lo, lo + 9)):
                col = e if e < nr else 2 * nr - 1 - e
                for par in (0, 1):
                    sg = -1.0 if par and e >= nr else 1.0
                    D1[par, j, col] += sg * w[t, 0]
                    D2[par, j, col] += sg * w[t, 1]
        xg, wg = np.polynomial.legendre.leggauss(nr)
        xg, wg, s = 0.5 * (xg + 1), 0.5 * wg, r ** 2
        W = np.array([0.5 * wg @ np.prod([(xg - s[i]) / (s[j] - s[i]) for i in range(nr) if i != j], axis=0)
                      for j in range(nr)])
        self.r = torch.tensor(r, **dev)
        self.W = torch.tensor(W, **dev)
        d1, d2 = torch.tensor(D1, **dev), torch.tensor(D2, **dev)
        m = torch.arange(-M, M + 1, device="cuda")
        self.m = m
        kz = 2.0 * math.pi / case["Lz"] * torch.arange(nk, **dev)
        self.ikz, self.imr = 1j * kz, 1j * m[:, None].double() / self.r  # [k], [m][j]
        self.What = 2.0 * math.pi * case["Lz"] * self.W[:, None, None] * torch.where(kz == 0, 1.0, 2.0)
        self.D1p, self.D1v = d1[m % 2], d1[(m + 1) % 2]  # [m][j][j'] for (p, u_z) and for (u_r, u_theta)
        mu = torch.arange(M + 2, device="cuda")
        L = d2[mu % 2] + d1[mu % 2] / self.r[:, None]
        eye = torch.eye(nr, **dev)
        L = L[:, None] - eye * ((mu[:, None, None, None].double() / self.r[:, None]) ** 2 + (kz ** 2)[None, :, None, None])
        A = eye / q["dt"] - L / (2 * q["Re"])
        A[:, :, 0] = eye[0]
        self.H = torch.linalg.inv(A)
        self.B = eye / q["dt"] + L / (2 * q["Re"])
        P = L[:M + 1].clone()
        P[:, :, 0] = d1[mu[:M + 1] % 2][:, None, 0]
        P[0, 0] = eye
        P = torch.linalg.inv(P)
        am = m.abs()
        self.P = P[am]
        self.Hm = [self.H[(m + 1).abs()], self.H[(m - 1).abs()], self.H[am]]
        self.Bm = [self.B[(m + 1).abs()], self.B[(m - 1).abs()], self.B[am]]
        # influence response to a unit wall datum, flux response of the mean mode
        phi = self.P[..., 0].to(torch.complex128)  # [m][k][j]
        h = self._helm(self._pm(-self._grad(phi)), None)
        h = torch.stack([(h[0] + h[1]) / 2, (h[0] - h[1]) / 2j, h[2]])
        delta = torch.einsum("mj,mkj->mk", self.D1v[:, 0].to(h.dtype), h[0])
        delta[M, 0] = 1.0
        h[:, M, 0] = 0.0
        self.infl = -h / delta[..., None]
        g = self.H[0, 0][:, 1:].sum(1)
        self.flux = g / (self.W @ g)
        kap = np.exp(0.75j * np.pi) * q["Wo"]
        J0, J1 = _bessel(0, kap), _bessel(1, kap)
        Bc = -0.5j * q["A"] / (1.0 - 2.0 * J1 / (kap * J0))
        self.Uh, self.dUh = Bc * (1.0 - _bessel(0, kap * r) / J0), Bc * kap * _bessel(1, kap * r) / J0
        self.rn = r

    # radial matrices act on the last axis; fields here are [m][k][j]
    @staticmethod
    def _mul(A, x):
        if A.dim() == 3:  # one matrix per m
            return torch.view_as_complex(torch.einsum("mij,mkjc->mkic", A, torch.view_as_real(x)).contiguous())
        return torch.view_as_complex(torch.matmul(A, torch.view_as_real(x)).contiguous())

    def _grad(self, p):
        return torch.stack([self._mul(self.D1p, p), self.imr[:, None] * p, self.ikz[:, None] * p])

    @staticmethod
    def _pm(f):
        return torch.stack([f[0] + 1j * f[1], f[0] - 1j * f[1], f[2]])

    def _helm(self, F, u):
        out = []
        for v in range(3):
            b = F[v] if u is None else F[v] + self._mul(self.Bm[v], u[v])
            b = torch.cat([torch.zeros_like(b[..., :1]), b[..., 1:]], -1)
            out.append(self._mul(self.Hm[v], b))
        return torch.stack(out)

    def _curl(self, u):
        imr, ikz = self.imr[:, None], self.ikz[:, None]
        return torch.stack([imr * u[2] - ikz * u[1], ikz * u[0] - self._mul(self.D1p, u[2]),
                            self._mul(self.D1v, u[1]) + u[1] / self.r - imr * u[0]])

    def _synth(self, f):  # [..][m][k][j] -> physical [..][j][theta][z]
        nr, M, K, nm, nk = self.dims
        f = f.movedim(-1, -3)
        x = torch.zeros(*f.shape[:-2], self.nt, self.nz // 2 + 1, dtype=f.dtype, device=f.device)
        x = torch.cat([torch.cat([f[..., M:, :], x[..., :self.nt - nm, :nk], f[..., :M, :]], -2),
                       x[..., nk:]], -1)
        return torch.fft.irfft(torch.fft.ifft(x, dim=-2, norm="forward"), self.nz, dim=-1, norm="forward")

    def _analyse(self, p):
        nr, M, K, nm, nk = self.dims
        x = torch.fft.fft(torch.fft.rfft(p, dim=-1, norm="forward")[..., :nk], dim=-2, norm="forward")
        return torch.cat([x[..., self.nt - M:, :], x[..., :M + 1, :]], -2).movedim(-3, -1)

    def _base(self, t):
        ph = np.exp(1j * self.q["Wo"] ** 2 / self.q["Re"] * t)
        U, dU = 1 - self.rn ** 2 + (self.Uh * ph).real, -2 * self.rn + (self.dUh * ph).real
        return torch.tensor(U, device="cuda"), torch.tensor(dU, device="cuda")

    def nonlinear(self, u, t):
        N = self._analyse(torch.linalg.cross(self._synth(u), self._synth(self._curl(u)), dim=0))
        U, dU = self._base(t)
        N = N - self.ikz[:, None] * U * u
        return torch.stack([N[0], N[1], N[2] - dU * u[0]])

    def nonlinear_adj(self, b, a, t):
        """Forcing of the continuous adjoint for w = b about the state a."""
        imr, ikz = self.imr[:, None], self.ikz[:, None]
        G = torch.stack([torch.stack([self._mul(self.D1v, a[0]), self._mul(self.D1v, a[1]), self._mul(self.D1p, a[2])]),
                         torch.stack([imr * a[0] - a[1] / self.r, imr * a[1] + a[0] / self.r, imr * a[2]]),
                         torch.stack([ikz * a[0], ikz * a[1], ikz * a[2]])])
        pa, pc, pb = self._synth(a), self._synth(self._curl(b)), self._synth(b)
        f = -torch.linalg.cross(pa, pc, dim=0)
        f = f - 2 * torch.stack([sum(self._synth(G[i, j]) * pb[j] for j in range(3)) for i in range(3)])
        U, dU = self._base(t)
        N = self._analyse(f) + ikz * U * b
        return torch.stack([N[0] - dU * b[2], N[1], N[2]])

    def stage(self, u, F):
        nr, M, K, nm, nk = self.dims
        div = self._mul(self.D1v, F[0]) + F[0] / self.r + self.imr[:, None] * F[1] + self.ikz[:, None] * F[2]
        keep = torch.ones(nm, nk, nr, device="cuda", dtype=torch.float64)
        keep[:, :, 0] = 0.0
        keep[M, 0] = 0.0
        p = self._mul(self.P, div * keep)
        x = self._helm(self._pm(F - self._grad(p)), self._pm(u))
        x = torch.stack([(x[0] + x[1]) / 2, (x[0] - x[1]) / 2j, x[2]])
        a0 = torch.einsum("mj,mkj->mk", self.D1v[:, 0].to(x.dtype), x[0])
        mean = torch.zeros(nm, nk, 1, device="cuda", dtype=torch.float64)
        mean[M, 0] = 1.0
        x = x + self.infl * a0[..., None]
        ur = x[0] * (1 - mean)
        uz = x[2] - mean * self.flux * (x[2] * self.W).sum(-1, keepdim=True)
        return torch.stack([ur, x[1], uz])

    def step(self, u, t):
        N0 = self.nonlinear(u, t)
        us = self.stage(u, N0)
        return self.stage(u, 0.5 * (N0 + self.nonlinear(us, t + self.q["dt"])))

    def step_adj(self, w, u_next, u_now, t_now):
        N0 = self.nonlinear_adj(w, u_next, t_now + self.q["dt"])
        ws = self.stage(w, N0)
        return self.stage(w, 0.5 * (N0 + self.nonlinear_adj(ws, u_now, t_now)))

    def pull(self, u, lam, t):
        """Euclidean cotangent of the step's input."""
        x = u.detach().requires_grad_(True)
        with torch.enable_grad():
            y = self.step(x, t)
        return torch.autograd.grad(y, x, lam)[0]


def _in(f):  # [c][j][m][k] -> [c][m][k][j]
    return f.permute(0, 2, 3, 1).contiguous()


def _out(f):
    return f.permute(0, 3, 1, 2).contiguous()


def _exact_gradient(p, u0, q, steps, continuous):
    energy = lambda v: 0.5 * float((p.What * _out(v).abs() ** 2).sum())  # noqa: E731
    u = _in(u0)
    u = u * math.sqrt(q["E0"] / energy(u))
    t = [q["tau0"] + n * q["dt"] for n in range(steps + 1)]
    states = [u]
    for n in range(steps):
        states.append(p.step(states[-1], t[n]))
    gain = energy(states[-1]) / q["E0"]
    if continuous:
        w = states[-1]
        for n in range(steps - 1, -1, -1):
            w = p.step_adj(w, states[n + 1], states[n], t[n])
        return _out(w), gain
    Wi = _in(p.What.expand(3, *p.What.shape[:1], p.dims[3], p.dims[4]))
    lam = Wi * states[-1]
    for n in range(steps - 1, -1, -1):
        lam = p.pull(states[n], lam, t[n])
    return _out(lam / Wi), gain


def exact(case, seed):
    requests, kind = _requests(case, seed), case["kind"]
    with torch.no_grad():
        if kind == "batch":
            got = [_exact_gradient(_Plain(case, q), _field(case, 100 * seed + i), q, case["steps"], False)
                   for i, q in enumerate(requests)]
            return {"gradient": [g for g, _ in got], "gain": np.array([e for _, e in got])}
        q = requests[0]
        p = _Plain(case, q)
        if kind == "forward":
            u = _in(_field(case, 100 * seed, _amplitude(case)))
            for n in range(case["steps"]):
                u = p.step(u, q["tau0"] + n * q["dt"])
            return {"u": _out(u)}
        if kind == "adjoint":
            Wi = _in(p.What.expand(3, *p.What.shape[:1], p.dims[3], p.dims[4]))
            u, lam = _in(_field(case, 100 * seed, _amplitude(case))), _in(_field(case, 100 * seed + 50, 1.0))
            return {"lam": _out(p.pull(u, Wi * lam, q["tau0"]) / Wi)}
        g, gain = _exact_gradient(p, _field(case, 100 * seed), q, case["steps"], kind == "continuous")
        return {"gradient": g, "gain": gain}
