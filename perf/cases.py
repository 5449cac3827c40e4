"""The work users of this package have it do, as timed cases.

Each case is one pass through the public entry points (``Solver``,
``AdiabaticSolver``): right-hand sides, runs of SSP-RK steps from a given
state, turbulence statistics and a training gradient of the learned sensor.
The meshes, degrees, precisions and options are those of the package's own
configurations (16^3 P1 FP64 driven to Mach 2; 64^3 P3 driven to Mach 3 in
FP32 and split-BF16 x3; 128^3 P2 driven to Mach 10; 128^3 P3 with the learned
sensor at Mach 6; 256^3 P3 decay; the two adiabatic workloads at 64^3) and of
its tests (ragged meshes, FP64 right-hand sides).

States are band-limited Gaussian random velocity fields with a k^-2 spectrum
and a density contrast, in the exact coefficients of their Fourier modes
cell by cell, made on the GPU from the seed.  A driven pass resumes from a
checkpoint (state and metadata), so that every pass does the same steps.

``exact`` is the method in plain torch in FP64: dense basis tables, the
quadrature sums as written in Sec. 2-3 of arXiv:2401.06841, and no code of
the package.
"""
import math

import numpy as np
import torch

CASES = [
    # the smallest mesh in use: 20 driven steps from rest in FP64, launch- and latency-bound
    dict(name="step_f64_k1_16", kind="iso", prec="f64", k=1, N=16, steps=20, mach=2.0, zeta=0.5, drive=True, rest=True,
         rk=2, riemann="rusanov", av="vnr"),
    # one FP64 right-hand side with a given driving: the parity mode (method studies)
    dict(name="rhs_f64_k3_24", kind="rhs", prec="f64", k=3, N=24, mach=2.0, drive=True, riemann="rusanov", av="vnr"),
    # one FP32 right-hand side on a ragged mesh (91125 cells) with the paper's face solver: time integrators of one's own
    dict(name="rhs_f32_k2_45", kind="rhs", prec="f32", k=2, N=45, mach=3.0, drive=True, riemann="hllc", av="vnr"),
    # Mach-3 driven turbulence, 64^3 P3, plain FP32: the everyday production run
    dict(name="step_f32_k3_64", kind="iso", prec="f32", k=3, N=64, steps=4, mach=3.0, zeta=0.5, drive=True, rest=False,
         rk=3, riemann="rusanov", av="vnr"),
    # the same run in the split-BF16 x3 mode
    dict(name="step_x3_k3_64", kind="iso", prec="x3", k=3, N=64, steps=4, mach=3.0, zeta=0.5, drive=True, rest=False,
         rk=3, riemann="rusanov", av="vnr"),
    # strong shocks: 128^3 P2, solenoidal driving to Mach 10, FP32
    dict(name="step_f32_k2_128", kind="iso", prec="f32", k=2, N=128, steps=2, mach=10.0, zeta=1.0, drive=True,
         rest=False, rk=3, riemann="rusanov", av="vnr"),
    # the learned viscosity sensor in a Mach-6 driven run, 128^3 P3, x3
    dict(name="learned_x3_k3_128", kind="iso", prec="x3", k=3, N=128, steps=2, mach=6.0, zeta=0.5, drive=True,
         rest=False, rk=3, riemann="rusanov", av="learned"),
    # the largest run: undriven decay at 256^3 P3, x3
    dict(name="step_x3_k3_256", kind="iso", prec="x3", k=3, N=256, steps=1, mach=3.0, zeta=0.5, drive=False, rest=False,
         rk=3, riemann="rusanov", av="vnr"),
    # decaying adiabatic turbulence, 64^3 P3 FP32
    dict(name="adi_f32_k3_64", kind="adi", prec="f32", k=3, N=64, steps=2, mach=0.5, gamma=1.4, drive=False, reset=False,
         riemann="rusanov"),
    # near-isothermal accounting: driven, temperature reset after every step, HLLC, 48^3 P2 FP32
    dict(name="adi_reset_f32_k2_48", kind="adi", prec="f32", k=2, N=48, steps=2, mach=1.0, gamma=1.0001, drive=True,
         reset=True, riemann="hllc"),
    # a training gradient of the learned sensor: one full batch of the P3 network
    dict(name="mlp_grad_k3_4096", kind="mlp", k=3, n=4096),
    # the statistics of a snapshot: density PDF, structure function, power spectrum, diagnostics
    dict(name="stats_f32_k3_64", kind="stats", prec="f32", k=3, N=64, mach=3.0, nbins=100, npairs=20000),
]


def listed():
    return [dict(c) for c in CASES]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: meshes over the logarithm of their range (odd ones among them), every degree, precision, face
    solver and sensor of the entry points above."""
    kind = rng.choice(["iso", "iso", "iso", "iso", "rhs", "adi", "adi"])
    k = rng.choice([1, 2, 3, 3])
    if kind == "rhs":
        prec = rng.choice(["f64", "f32", "f32"])
        hi = {"f64": {1: 64, 2: 48, 3: 36}, "f32": {1: 128, 2: 96, 3: 80}}[prec][k]
        return dict(kind="rhs", prec=prec, k=k, N=_log_int(rng, 8, hi), mach=rng.choice([1.0, 2.0, 3.0]),
                    drive=rng.random() < 0.5, riemann=rng.choice(["rusanov", "hll", "hllc"]),
                    av=rng.choice(["vnr", "vnr", "off"]))
    if kind == "adi":
        reset = rng.random() < 0.4
        return dict(kind="adi", prec="f32", k=k, N=_log_int(rng, 12, {1: 112, 2: 88, 3: 72}[k]),
                    steps=rng.choice([1, 2, 3]), mach=1.0 if reset else 0.5, gamma=1.0001 if reset else 1.4,
                    drive=reset, reset=reset, riemann=rng.choice(["rusanov", "hllc"]))
    prec = rng.choice(["f64", "f32", "f32", "f32", "x3", "x3", "x3"])
    hi = {1: 160, 2: 128, 3: 112} if prec != "f64" else {1: 48, 2: 32, 3: 24}
    return dict(kind="iso", prec=prec, k=k, N=_log_int(rng, 8 if prec == "f64" else 12, hi[k]),
                steps=rng.choice([1, 2, 3, 4]), mach=rng.choice([1.0, 2.0, 3.0, 6.0]), zeta=rng.choice([0.5, 1.0]),
                drive=rng.random() < 0.5, rest=False, rk=2 if k == 1 else rng.choice([2, 3, 3]),
                riemann=rng.choice(["rusanov", "rusanov", "hll", "hllc"]),
                av=rng.choice(["vnr", "vnr", "vnr", "off", "learned"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _modes(k):
    return [(i, j, d - i - j) for d in range(k + 1) for i in range(d, -1, -1) for j in range(d - i, -1, -1)]


def _spherical_jn(m, a):
    """j_m(a), m <= 3, |a| <= pi/4 here: the power series."""
    s, t = torch.zeros_like(a), torch.ones_like(a)
    for j in range(14):
        den = 1.0
        for q in range(1, 2 * j + 2 * m + 2, 2):
            den *= q
        num = 1.0
        for q in range(1, 2 * j, 2):
            num *= q
        # a^m sum_j (-a^2/2)^j / (j! (2m+2j+1)!!)
        s = s + t / (math.factorial(j) * den)
        t = t * (-a * a / 2)
    return a ** m * s


def _field(N, k, gen, ncomp, zeta, dtype, dev):
    """[N^3][ncomp][b] coefficients of a random field with shell spectrum E(k) ~ k^-2 on 2 <= |k| <= max(2, N/4), rms 1
    in its cell means (ncomp = 3: Helmholtz-mixed with solenoidal weight zeta)."""
    f64 = torch.float64
    kk = torch.fft.fftfreq(N, d=1.0 / N, device=dev, dtype=f64)
    KZ, KY, KX = torch.meshgrid(kk, kk, kk, indexing="ij")
    K = torch.sqrt(KX ** 2 + KY ** 2 + KZ ** 2)
    band = (K >= 2) & (K <= max(2.0, N / 4))
    Ks = torch.where(K > 0, K, torch.ones_like(K))
    amp = torch.where(band, Ks ** -2.0, torch.zeros_like(K))
    A = [torch.complex(torch.randn(K.shape, generator=gen, device=dev, dtype=f64),
                       torch.randn(K.shape, generator=gen, device=dev, dtype=f64)) * amp for _ in range(ncomp)]
    if ncomp == 3:
        kh = [KX / Ks, KY / Ks, KZ / Ks]
        dot = sum(h * a for h, a in zip(kh, A))
        A = [zeta * (a - h * dot) + (1 - zeta) * h * dot for h, a in zip(kh, A)]
        del kh, dot
    del KX, KY, KZ, K, Ks, amp, band
    h = 1.0 / N
    # per axis: sqrt(2m+1) i^m j_m(pi kappa h) exp(i pi kappa / N)
    ph = torch.polar(torch.ones_like(kk), math.pi * kk / N)
    g = [math.sqrt(2 * m + 1) * (1j ** m) * _spherical_jn(m, math.pi * kk * h) * ph for m in range(k + 1)]
    out = torch.empty(N ** 3, ncomp, len(_modes(k)), dtype=dtype, device=dev)
    rms2 = 0.0
    for l, (i, j, z) in enumerate(_modes(k)):
        G = g[z][:, None, None] * g[j][None, :, None] * g[i][None, None, :]
        for c in range(ncomp):
            f = torch.fft.ifftn(A[c] * G).real.reshape(-1) * float(N) ** 3
            if l == 0:
                rms2 = rms2 + (f ** 2).mean()
            out[:, c, l] = f.to(dtype)
    out *= float(1.0 / torch.sqrt(rms2))
    return out


def _dtype(case):
    return torch.float64 if case.get("prec") == "f64" else torch.float32


def _state(case, seed, dev):
    """The case's initial coefficients [N^3][4 or 5][b] in its element type."""
    N, k, dt = case["N"], case["k"], _dtype(case)
    b = len(_modes(k))
    nv = 5 if case["kind"] == "adi" else 4
    if case.get("rest"):
        u = torch.zeros(N ** 3, nv, b, dtype=dt, device=dev)
        u[:, 0, 0] = 1.0
        return u
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    u = torch.empty(N ** 3, nv, b, dtype=dt, device=dev)
    u[:, 1:4] = _field(N, k, gen, 3, case.get("zeta", 0.5), dt, dev)
    cs = math.sqrt(case["gamma"]) if nv == 5 and not case["reset"] else 1.0
    u[:, 1:4] *= case["mach"] * cs
    rho = _field(N, k, gen, 1, 0.0, dt, dev)
    u[:, 0] = rho[:, 0] * (0.12 if nv == 4 else 0.06)
    u[:, 0, 0] += 1.0
    if nv == 5:
        # total energy: unit mean pressure (or, with the reset, the offset energy of the uniform temperature) plus the
        # kinetic energy of the cell means
        u[:, 4] = 0.0
        u[:, 4, 0] = 0.5 * (u[:, 1:4, 0] ** 2).sum(dim=1) / u[:, 0, 0]
        if not case["reset"]:
            u[:, 4, 0] += 1.0 / (case["gamma"] - 1.0)
    return u


def _ahat(case, seed, dev):
    """A given driving [N^3][3][b]: a smooth random acceleration of order 2 Mach^2."""
    gen = torch.Generator(device=dev).manual_seed(int(seed) + 1000003)
    return _field(case["N"], case["k"], gen, 3, 0.5, _dtype(case), dev) * (2.0 * case["mach"] ** 2)


def _weights(k, seed):
    """Seeded parameters of the sensor network, layout W1 [64][D], b1, W2 [64][64], b2, W3, b3: Kaiming-uniform, the
    last layer narrowed so that nu/(cs h/p) = exp(y) lies around one half."""
    D, H = 2 * len(_modes(k)), 64
    rng = np.random.default_rng(int(seed) + 77)
    w1 = rng.uniform(-1, 1, H * D) * math.sqrt(6.0 / D)
    w2 = rng.uniform(-1, 1, H * H) * math.sqrt(6.0 / H)
    w3 = 0.3 * rng.uniform(-1, 1, H) * math.sqrt(6.0 / H)
    return np.concatenate([w1, np.zeros(H), w2, np.zeros(H), w3, [math.log(0.5)]]).astype(np.float32)


def _pairs(case, seed, dev):
    """Training pairs with the sensor's input layout: rho_l/rho_0 and the projected |v|/cs, and log-coefficients."""
    k, n = case["k"], case["n"]
    b = len(_modes(k))
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    deg = torch.tensor([sum(m) for m in _modes(k)], device=dev, dtype=torch.float32)
    x = torch.randn(n, 2 * b, generator=gen, device=dev)
    x[:, :b] *= 0.3 * 0.5 ** deg
    x[:, 0] = 1.0
    x[:, b:] *= 0.6 * 0.5 ** deg
    x[:, b] = x[:, b].abs() + 2.0
    y = torch.log(0.2 + (x[:, 1:4].abs().sum(dim=1) + 0.3 * x[:, b + 1:b + 4].abs().sum(dim=1)))
    return x.contiguous(), y.contiguous()


def prepare(case, seed):
    from paper_2401_06841_gb300 import AdiabaticSolver, Solver
    dev = torch.device("cuda", torch.cuda.current_device())
    kind = case["kind"]
    st = {"case": case}
    if kind == "adi":
        s = AdiabaticSolver(case["N"], case["k"], gamma=case["gamma"], precision=case["prec"], riemann=case["riemann"])
        if case["reset"]:
            s.set_reset(1.0)
        if case["drive"]:
            s.set_forcing(mach=case["mach"], zeta=0.5, seed=int(seed), cs_ref=1.0)
        st["meta"] = s.get_meta()
        st["u"] = _state(case, seed, dev)
    elif kind == "mlp":
        s = Solver(4, case["k"], precision="f32", av="learned")
        s.set_av_weights(_weights(case["k"], seed))
        st["x"], st["y"] = _pairs(case, seed, dev)
    else:
        s = Solver(case["N"], case["k"], precision=case["prec"], rk_stages=case.get("rk"),
                   riemann=case.get("riemann", "rusanov"), av=case.get("av", "vnr"))
        if case.get("av") == "learned":
            s.set_av_weights(_weights(case["k"], seed))
        if kind == "iso" and case["drive"]:
            s.set_forcing(mach=case["mach"], zeta=case["zeta"], seed=int(seed))
        st["meta"] = s.get_meta()
        st["u"] = _state(case, seed, dev)
        if kind == "rhs" and case["drive"]:
            st["a"] = _ahat(case, seed, dev)
        if kind == "stats":
            s.set_state(st["u"])
    st["s"] = s
    return st


def _dt_pimax(case):
    return 0.05 / (case["N"] * (case["k"] + 1))


def run(state):
    case, s = state["case"], state["s"]
    kind = case["kind"]
    if kind in ("iso", "adi"):
        # resume from a checkpoint, advance, take the new state
        s.set_state(state["u"])
        s.set_meta(state["meta"])
        t, dt = s.step(case["steps"])
        return {"u": s.get_state(), "t": t, "dt": dt}
    if kind == "rhs":
        return {"dudt": s.rhs(state["u"], ahat=state.get("a"), dt_pimax=_dt_pimax(case))}
    if kind == "mlp":
        loss, grad = s.mlp_grad(state["x"], state["y"])
        return {"loss": loss, "grad": grad}
    hist = s.density_pdf(nbins=200)
    l, v = s.structure_function(nbins=case["nbins"], npairs=case["npairs"], seed=1)
    kmean, power, count = s.power_spectrum()
    d = s.diagnostics()
    return {"hist": hist, "l": l, "v": v, "kmean": kmean, "power": power, "count": count,
            "diag": np.array([d[n] for n in ("mass", "ekin", "mach", "mach_rho", "rho_min", "rho_max", "max_speed")])}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    k = case["k"]
    b, n = len(_modes(k)), k + 1
    if case["kind"] == "mlp":
        P = 64 * 2 * b + 64 * 64 + 3 * 64 + 1
        rows = case["n"]
        return {"bytes": 4.0 * (rows * (2 * b + 1) + 2 * P), "flops": 6.0 * rows * (64 * 2 * b + 64 * 64 + 64)}
    N, e = case["N"], 8 if case["prec"] == "f64" else 4
    nc, p2 = N ** 3, (k + 1) * (k + 2) // 2
    vol = b * n + p2 * n * n + n ** 4           # multiply-adds: one field to or from the Gauss points, axis by axis
    face = b + p2 * n + n ** 3                  # one field to or from the points of a face
    if case["kind"] == "stats":
        g = float((n * N) ** 3)
        return {"bytes": e * nc * 4.0 * b, "flops": 2.0 * 4 * vol * nc + 3 * 2.5 * g * math.log2(g)
                + 2.0 * 2 * 4 * b * case["nbins"] * case["npairs"]}
    nv = 5 if case["kind"] == "adi" else 4
    drive = 3 if case["drive"] else 0
    # per cell: the fields, grad rho and div m at the points; fluxes, primitives and the source back; three faces
    mul = vol * (nv + 4 + drive) + vol * (6 + 3 * (nv - 4) + (nv - 1) + drive * (nv - 3)) + 3 * face * nv * 4
    flops = nc * (2.0 * mul + 60 * n ** 3 + 3 * 40 * n * n)
    words = nc * float(b)
    if case["kind"] == "rhs":
        return {"bytes": e * words * (2 * nv + drive), "flops": flops}
    rk = case.get("rk") or (2 if k == 1 else 3)
    per_step = rk * 2 * nv + (rk - 1) * nv + rk * drive
    return {"bytes": e * words * per_step * case["steps"], "flops": flops * rk * case["steps"]}


# ---------------------------------------------------------------------------
# the same in plain torch, FP64
# ---------------------------------------------------------------------------
class _Ref:
    def __init__(self, case, dev):
        f64 = torch.float64
        self.N, self.k, self.dev = case["N"], case["k"], dev
        self.h = 1.0 / self.N
        self.hp = self.h / (self.k + 1)
        n = self.k + 1
        x, w = np.polynomial.legendre.leggauss(n)

        def pn(m, t):
            return math.sqrt(2 * m + 1) * np.polynomial.legendre.legval(t, [0] * m + [1])

        def dpn(m, t):
            return math.sqrt(2 * m + 1) * np.polynomial.legendre.legval(
                t, np.polynomial.legendre.legder(np.array([0.0] * m + [1.0])))

        P = np.array([pn(m, x) for m in range(n)])
        D = np.array([dpn(m, x) + 0 * x for m in range(n)])
        E = [np.array([pn(m, s) for m in range(n)]) for s in (-1.0, 1.0)]
        md = _modes(self.k)
        self.b, self.md, self.x1, self.w1, self.P = len(md), md, x, w, P
        vol = lambda A, B, C: np.stack([np.einsum("a,b,c->cba", A[i], B[j], C[z]).ravel() for i, j, z in md])  # noqa: E731
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=f64, device=dev)  # noqa: E731
        self.phi = T(vol(P, P, P))                                     # [b][nq]
        self.dphi = [T(vol(D, P, P)), T(vol(P, D, P)), T(vol(P, P, D))]
        self.wq = T(np.einsum("a,b,c->cba", w, w, w).ravel() / 8)
        self.phif = []
        for d in range(3):
            t = [a for a in range(3) if a != d]
            self.phif.append([T(np.stack([E[s][m[d]] * np.einsum("a,c->ca", P[m[t[0]]], P[m[t[1]]]).ravel()
                                          for m in md])) for s in (0, 1)])
        self.ws = T(np.einsum("a,c->ca", w, w).ravel())

    def roll(self, f, d):
        """f of the neighbour across the + face along d."""
        N = self.N
        return torch.roll(f.reshape((N, N, N) + f.shape[1:]), -1, dims=2 - d).reshape(f.shape)

    def roll_back(self, f, d):
        N = self.N
        return torch.roll(f.reshape((N, N, N) + f.shape[1:]), 1, dims=2 - d).reshape(f.shape)

    def back(self, f):
        """Gauss projection of point values [..., nq] onto the basis."""
        return (f * self.wq) @ self.phi.T

    def chunks(self, n):
        step = max(1, (1 << 25) // (self.phi.shape[1] * 8))
        return [slice(i, min(n, i + step)) for i in range(0, n, step)]

    # -- isothermal -----------------------------------------------------
    def project(self, u):
        out = torch.empty(u.shape[0], 3, self.b, dtype=u.dtype, device=u.device)
        vabs = torch.empty(u.shape[0], self.b, dtype=u.dtype, device=u.device)
        smax = 0.0
        for s in self.chunks(u.shape[0]):
            f = u[s] @ self.phi
            v = f[:, 1:] / f[:, :1]
            out[s] = self.back(v)
            vabs[s] = self.back(v.square().sum(dim=1).sqrt())
            smax = max(smax, float(v.abs().sum(dim=1).max()) + 3.0)
        return out, vabs, smax

    def abar(self, u, a):
        return (u[:, 0, None] * a).sum(dim=(0, 2)) / u[:, 0, 0].sum()

    def flux(self, W, d):
        rho, v = W[:, 0], W[:, 1:4]
        F = torch.cat([(rho * v[:, d])[:, None], rho[:, None] * v * v[:, d:d + 1]], dim=1)
        F[:, 1 + d] += rho
        return F

    def riemann(self, kind, L, R, d):
        UL = torch.cat([L[:, :1], L[:, :1] * L[:, 1:]], dim=1)
        UR = torch.cat([R[:, :1], R[:, :1] * R[:, 1:]], dim=1)
        FL, FR = self.flux(L, d), self.flux(R, d)
        vl, vr = L[:, 1 + d], R[:, 1 + d]
        if kind == "rusanov":
            lam = torch.maximum(vl.abs(), vr.abs()) + 1.0
            return 0.5 * (FL + FR) - 0.5 * lam[:, None] * (UR - UL)
        SL, SR = torch.minimum(vl, vr) - 1.0, torch.maximum(vl, vr) + 1.0
        inv = 1.0 / (SR - SL)
        F = (SR[:, None] * FL - SL[:, None] * FR + (SL * SR)[:, None] * (UR - UL)) * inv[:, None]
        if kind == "hllc":
            rs = (SR * UR[:, 0] - SL * UL[:, 0] - (FR[:, 0] - FL[:, 0])) * inv
            ms = (SR * UR[:, 1 + d] - SL * UL[:, 1 + d] - (FR[:, 1 + d] - FL[:, 1 + d])) * inv
            up = torch.where((ms / rs >= 0)[:, None], L, R)
            for t in range(3):
                if t != d:
                    F[:, 1 + t] = F[:, 0] * up[:, 1 + t]
        F = torch.where((SL >= 0)[:, None], FL, F)
        return torch.where((SR <= 0)[:, None], FR, F)

    def faces(self, R, W, solver):
        """Adds the surface terms of the face states W [c][fields][b]."""
        i4h = 0.25 / self.h
        for d in range(3):
            F = solver(W @ self.phif[d][1], self.roll(W, d) @ self.phif[d][0], d) * self.ws
            R -= i4h * (F @ self.phif[d][1].T)
            R += i4h * (self.roll_back(F, d) @ self.phif[d][0].T)

    def rhs(self, u, kind, av, dt, a=None, nu=None):
        c2 = 2.0 / self.h
        vh, _, _ = self.project(u)
        ab = self.abar(u, a) if a is not None else None
        R = torch.empty_like(u)
        for s in self.chunks(u.shape[0]):
            f = u[s] @ self.phi
            rho, m = f[:, 0], f[:, 1:]
            v = m / rho[:, None]
            Pi = torch.zeros_like(rho)
            if av != "off":
                gr = [c2 * (u[s, 0] @ D) for D in self.dphi]
                dm = sum(c2 * (u[s, 1 + d] @ self.dphi[d]) for d in range(3))
                D = (dm - sum(v[:, d] * gr[d] for d in range(3))) / rho
                A = (-D).clamp(min=0.0)
                Pi = (2.0 * rho * self.hp ** 2 * A * A + 0.2 * rho * self.hp * A) if nu is None else rho * nu[s, None] * A
                if dt > 0:
                    Pi = torch.minimum(Pi, rho * self.hp ** 2 * A / (2 * dt))
            r = 0.0
            for d in range(3):
                F = torch.cat([m[:, d:d + 1], m * v[:, d:d + 1]], dim=1)
                F[:, 1 + d] += rho + Pi
                r = r + c2 * ((F * self.wq) @ self.dphi[d].T)
            if a is not None:
                acc = a[s] @ self.phi - ab[None, :, None]
                r[:, 1:] += self.back(rho[:, None] * acc)
            R[s] = r
        self.faces(R, torch.cat([u[:, :1], vh], dim=1), lambda L, Rr, d: self.riemann(kind, L, Rr, d))
        return R

    def limit(self, u, eps=1e-3):
        """The density floor at the volume and face points; None where a mean is at the floor."""
        pts = torch.cat([self.phi] + [t for d in self.phif for t in d], dim=1)
        mn = torch.cat([(u[s, 0] @ pts).amin(dim=1) for s in self.chunks(u.shape[0])])
        low = mn < eps
        if not bool(low.any()):
            return u
        if bool((u[low, 0, 0] <= eps).any()):
            return None
        th = torch.where(low, (u[:, 0, 0] - eps) / torch.where(low, u[:, 0, 0] - mn, torch.ones_like(mn)),
                         torch.ones_like(mn))
        u[:, :, 1:] *= th[:, None, None]
        return u

    def sensor(self, u, k, w):
        _, vabs, _ = self.project(u)
        y = _net(torch.cat([u[:, 0] / u[:, 0, :1], vabs], dim=1), w)
        return self.hp * torch.exp(y)

    # -- adiabatic ------------------------------------------------------
    def adi_project(self, u, g):
        out = torch.empty(u.shape[0], 4, self.b, dtype=u.dtype, device=u.device)
        smax, pmin, rmin = 0.0, 1e300, 1e300
        for s in self.chunks(u.shape[0]):
            f = u[s] @ self.phi
            v = f[:, 1:4] / f[:, :1]
            p = (g - 1) * (f[:, 4] - 0.5 * (f[:, 1:4] * v).sum(dim=1))
            out[s, :3], out[s, 3] = self.back(v), self.back(p)
            smax = max(smax, float((v.abs().sum(dim=1) + 3 * (g * p / f[:, 0]).sqrt()).max()))
            pmin, rmin = min(pmin, float(p.min())), min(rmin, float(f[:, 0].min()))
        return out, smax, min(pmin, rmin)

    def adi_cons(self, W, g):
        rho, v, p = W[:, 0], W[:, 1:4], W[:, 4]
        return torch.cat([rho[:, None], rho[:, None] * v,
                          (p / (g - 1) + 0.5 * rho * v.square().sum(dim=1))[:, None]], dim=1)

    def adi_flux(self, W, U, d):
        vn, p = W[:, 1 + d], W[:, 4]
        F = U * vn[:, None]
        F[:, 1 + d] += p
        F[:, 4] += p * vn
        return F

    def adi_riemann(self, kind, L, R, d, g):
        UL, UR = self.adi_cons(L, g), self.adi_cons(R, g)
        FL, FR = self.adi_flux(L, UL, d), self.adi_flux(R, UR, d)
        ul, ur = L[:, 1 + d], R[:, 1 + d]
        cl, cr = (g * L[:, 4] / L[:, 0]).sqrt(), (g * R[:, 4] / R[:, 0]).sqrt()
        if kind == "rusanov":
            lam = torch.maximum(ul.abs() + cl, ur.abs() + cr)
            return 0.5 * (FL + FR) - 0.5 * lam[:, None] * (UR - UL)
        SL, SR = torch.minimum(ul - cl, ur - cr), torch.maximum(ul + cl, ur + cr)
        qL, qR = L[:, 0] * (SL - ul), R[:, 0] * (SR - ur)
        Ss = (R[:, 4] - L[:, 4] + ul * qL - ur * qR) / (qL - qR)
        lft = Ss >= 0
        pick = lambda a, c: torch.where(lft if a.dim() == 2 else lft[:, None], a, c)  # noqa: E731
        SK, qK, uK, W, U, F = pick(SL, SR), pick(qL, qR), pick(ul, ur), pick(L, R), pick(UL, UR), pick(FL, FR)
        f = qK / (SK - Ss)
        Us = torch.cat([f[:, None], f[:, None] * W[:, 1:4],
                        (f * (U[:, 4] / W[:, 0] + (Ss - uK) * (Ss + W[:, 4] / qK)))[:, None]], dim=1)
        Us[:, 1 + d] = f * Ss
        F = F + SK[:, None] * (Us - U)
        F = torch.where((SL >= 0)[:, None], FL, F)
        return torch.where((SR <= 0)[:, None], FR, F)

    def adi_rhs(self, u, g, kind, dt, a=None):
        c2 = 2.0 / self.h
        pr, _, _ = self.adi_project(u, g)
        ab = self.abar(u, a) if a is not None else None
        R = torch.empty_like(u)
        for s in self.chunks(u.shape[0]):
            f = u[s] @ self.phi
            rho, m, e = f[:, 0], f[:, 1:4], f[:, 4]
            v = m / rho[:, None]
            p = (g - 1) * (e - 0.5 * (m * v).sum(dim=1))
            gr = [c2 * (u[s, 0] @ D) for D in self.dphi]
            dm = sum(c2 * (u[s, 1 + d] @ self.dphi[d]) for d in range(3))
            A = (-(dm - sum(v[:, d] * gr[d] for d in range(3))) / rho).clamp(min=0.0)
            Pi = 2.0 * rho * self.hp ** 2 * A * A + 0.2 * rho * (g * p / rho).sqrt() * self.hp * A
            if dt > 0:
                Pi = torch.minimum(Pi, rho * self.hp ** 2 * A / (2 * dt))
            P = p + Pi
            r = 0.0
            for d in range(3):
                F = f * v[:, d:d + 1]
                F[:, 1 + d] += P
                F[:, 4] += P * v[:, d]
                r = r + c2 * ((F * self.wq) @ self.dphi[d].T)
            if a is not None:
                acc = a[s] @ self.phi - ab[None, :, None]
                r[:, 1:4] += self.back(rho[:, None] * acc)
                r[:, 4] += self.back((m * acc).sum(dim=1))
            R[s] = r
        self.faces(R, torch.cat([u[:, :1], pr], dim=1), lambda L, Rr, d: self.adi_riemann(kind, L, Rr, d, g))
        return R

    # -- driving (Sec. 4.2) ---------------------------------------------
    def accel(self, kv, amp):
        """Gauss projection [N^3][3][b] of sum_m 2 Re(amp_m exp(2 pi i k_m.x)), axis by axis."""
        N, n = self.N, self.k + 1
        i = np.arange(N)[:, None]
        xs = (i + 0.5 + 0.5 * self.x1[None, :]) * self.h
        G = {}
        for q in range(-8, 9):
            e = np.exp(2j * np.pi * q * xs)
            G[q] = torch.as_tensor(np.einsum("ia,a,ma->im", e, self.w1 / 2, self.P), device=self.dev)
        out = torch.zeros(N ** 3, 3, self.b, dtype=torch.float64, device=self.dev)
        ix, iy, iz = (torch.tensor([m[d] for m in self.md], device=self.dev) for d in range(3))
        for (kx, ky, kz), am in zip(kv, amp):
            g = (G[kz][:, None, None, iz] * G[ky][None, :, None, iy] * G[kx][None, None, :, ix]).reshape(N ** 3, self.b)
            for c in range(3):
                out[:, c] += 2 * (g.real * am[c].real - g.imag * am[c].imag)
        return out


class _OU:
    """The Ornstein-Uhlenbeck driving with SplitMix64 and Box-Muller draws, modes 1 <= |k|^2 <= 9, cs = 1."""

    def __init__(self, mach, zeta, seed):
        self.kv = [(a, b, c) for a in range(-3, 4) for b in range(-3, 4) for c in range(-3, 4)
                   if 1 <= a * a + b * b + c * c <= 9 and (a or b or c) > 0]
        self.zeta, self.rng, self.spare = zeta, int(seed) & (2 ** 64 - 1), None
        tc = 1.0 / (2.0 * mach)
        self.dtd = self.t_next = tc / 100.0
        self.f = math.exp(-self.dtd / tc)
        self.s = 2.0 * mach ** 2 / math.sqrt(4.0 * len(self.kv) * (2 * zeta ** 2 + (1 - zeta) ** 2))
        self.x = [[[self.s * self.normal() for _ in range(2)] for _ in range(3)] for _ in self.kv]

    def uni(self):
        M = 2 ** 64 - 1
        self.rng = (self.rng + 0x9E3779B97F4A7C15) & M
        z = self.rng
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M
        return ((z ^ (z >> 31)) >> 11) * 2.0 ** -53

    def normal(self):
        if self.spare is not None:
            v, self.spare = self.spare, None
            return v
        u1 = 1.0 - self.uni()
        u2 = self.uni()
        r, ang = math.sqrt(-2.0 * math.log(u1)), 2.0 * math.pi * u2
        self.spare = r * math.sin(ang)
        return r * math.cos(ang)

    def advance(self):
        c = self.s * math.sqrt(1.0 - self.f ** 2)
        self.x = [[[self.f * q + c * self.normal() for q in p] for p in m] for m in self.x]

    def amplitudes(self):
        out = []
        for kv, x in zip(self.kv, self.x):
            k = np.array(kv, dtype=np.float64)
            L = np.outer(k, k) / (k @ k)
            z = np.array([p[0] + 1j * p[1] for p in x])
            out.append(((self.zeta * (np.eye(3) - L) + (1 - self.zeta) * L) @ z).tolist())
        return out


def _net(x, w):
    """The sensor network in FP64."""
    D, H = x.shape[1], 64
    w = torch.as_tensor(np.asarray(w), dtype=torch.float64, device=x.device) if not torch.is_tensor(w) else w
    W1, r = w[:H * D].reshape(H, D), w[H * D:]
    b1, W2, b2, W3, b3 = r[:H], r[H:H + H * H].reshape(H, H), r[H + H * H:2 * H + H * H], r[-H - 1:-1], r[-1]
    z = torch.nn.functional.gelu(x @ W1.T + b1)
    z = torch.nn.functional.gelu(z @ W2.T + b2)
    return z @ W3 + b3


_RK = {2: [(0.0, 1.0), (0.5, 0.5)], 3: [(0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)]}


def _exact_steps(case, seed, dev):
    N, k, adi = case["N"], case["k"], case["kind"] == "adi"
    ref = _Ref(case, dev)
    u = _state(case, seed, dev).double()
    rk = _RK[case.get("rk") or (2 if k == 1 else 3)]
    drv = _OU(case["mach"], case.get("zeta", 0.5), seed) if case["drive"] else None
    g = case.get("gamma")
    kap = 1.0 / (g - 1) if adi and case["reset"] else 0.0
    if adi:
        u[:, 4] += kap * u[:, 0]
    t, dt, a = 0.0, 0.0, None
    for _ in range(case["steps"]):
        if drv:
            new = a is None
            while t >= drv.t_next:
                drv.advance()
                drv.t_next += drv.dtd
                new = True
            if new:
                a = ref.accel(drv.kv, drv.amplitudes())
        if adi:
            _, smax, low = ref.adi_project(u, g)
            if not low > 2e-3:
                return None
        else:
            _, _, smax = ref.project(u)
        nu = ref.sensor(u, k, _weights(k, seed)) if case.get("av") == "learned" else None
        dt = 0.3 * ref.h / ((k + 1) * smax)
        v = u
        for ra, rb in rk:
            r = ref.adi_rhs(v, g, case["riemann"], dt, a) if adi else ref.rhs(v, case["riemann"], case["av"], dt, a, nu)
            v = rb * (v + dt * r) + (ra * u if ra else 0.0)
            if not adi:
                v = ref.limit(v)
                if v is None:
                    return None
        u = v
        t += dt
        if adi and case["reset"]:
            for s in ref.chunks(u.shape[0]):
                f = u[s, :4] @ ref.phi
                u[s, 4] = ref.back(0.5 * f[:, 1:4].square().sum(dim=1) / f[:, 0]) + kap * u[s, 0]
    if adi:
        u[:, 4] -= kap * u[:, 0]
    return {"u": u, "t": t, "dt": dt}


def _exact_stats(case, seed, dev):
    ref = _Ref(case, dev)
    u = _state(case, seed, dev).double()
    N, n = case["N"], case["k"] + 1
    f = torch.cat([u[s] @ ref.phi for s in ref.chunks(u.shape[0])])
    rho, v = f[:, 0], f[:, 1:] / f[:, :1]
    w = ref.wq / N ** 3
    mean = float(u[:, 0, 0].mean())
    bins = torch.floor((torch.log10(rho / mean) + 2.0) / (4.0 / 200)).long()
    ok = (bins >= 0) & (bins < 200)
    hist = torch.zeros(200, dtype=torch.float64, device=dev)
    hist.index_add_(0, bins[ok], w.expand_as(rho)[ok])
    ekin = float((0.5 * (f[:, 1:] * v).sum(dim=1) * w).sum())
    v2 = v.square().sum(dim=1)
    diag = [mean, ekin, math.sqrt(float((v2 * w).sum())), math.sqrt(2 * ekin / mean), float(rho.min()),
            float(rho.max()), float(v.abs().sum(dim=1).max()) + 3.0]
    # the velocity at x_g = (g + 1/2)/Ng, its transform and the shell sums
    Ng, nb = n * N, 2000
    xg = (2 * np.arange(n) + 1) / n - 1
    Pg = [math.sqrt(2 * m + 1) * np.polynomial.legendre.legval(xg, [0] * m + [1]) for m in range(n)]
    T = torch.as_tensor(np.stack([np.einsum("a,b,c->cba", Pg[i], Pg[j], Pg[z]).ravel() for i, j, z in ref.md]),
                        device=dev)
    fg = torch.cat([u[s] @ T for s in ref.chunks(u.shape[0])])
    kk = torch.fft.fftfreq(Ng, d=1.0 / Ng, device=dev, dtype=torch.float64)
    K2 = kk[:, None, None] ** 2 + kk[None, :, None] ** 2 + kk[None, None, :] ** 2
    K = K2.sqrt().reshape(-1)
    nz = K > 0
    shell = torch.floor(torch.log(K[nz]) / math.log(math.sqrt(3.0) * Ng / 2) * nb).long().clamp(max=nb - 1)
    power, ksum, count = (torch.zeros(nb, dtype=torch.float64, device=dev) for _ in range(3))
    ksum.index_add_(0, shell, K[nz])
    count.index_add_(0, shell, torch.ones_like(K[nz]))
    for d in range(3):
        x = (fg[:, 1 + d] / fg[:, 0]).reshape(N, N, N, n, n, n).permute(0, 3, 1, 4, 2, 5).reshape(Ng, Ng, Ng)
        F = torch.fft.fftn(x) / float(Ng) ** 3
        power.index_add_(0, shell, (F.real.square() + F.imag.square()).reshape(-1)[nz])
    kmean = torch.where(count > 0, ksum / count.clamp(min=1), torch.zeros_like(ksum))
    return {"hist": hist, "l": None, "v": None, "kmean": kmean, "power": power, "count": None, "diag": np.array(diag)}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind = case["kind"]
    if kind == "mlp":
        x, y = _pairs(case, seed, dev)
        w = torch.tensor(_weights(case["k"], seed), dtype=torch.float64, device=dev, requires_grad=True)
        loss = (_net(x.double(), w) - y.double()).square().mean()
        loss.backward()
        return {"loss": loss.item(), "grad": w.grad}
    if case["N"] > 160:  # minutes
        return None
    if kind == "stats":
        return _exact_stats(case, seed, dev)
    if kind == "rhs":
        ref = _Ref(case, dev)
        a = _ahat(case, seed, dev).double() if case["drive"] else None
        return {"dudt": ref.rhs(_state(case, seed, dev).double(), case["riemann"], case["av"], _dt_pimax(case), a)}
    return _exact_steps(case, seed, dev)
