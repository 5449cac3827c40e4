"""The kernels at the sizes where their tilings can go wrong: meshes below, at and
just past a brick (4 x 4 x 2 cells), a block of 32 cells and a tile of 64, all
degrees, face solvers and element types, result buffers that no vector store may
touch, driving modes in every order and sign, training batches around a block of 32
samples, statistics on grids with and without a Nyquist plane, and runs of steps
against single steps.  The reference is the FP64 oracle on the same inputs.

Bounds (relative L2 per field): one evaluation in FP64 1e-12 and in FP32 1e-5, as
in test_gpu_parity.py (unit round-off times the cancellation in the flux
divergence); the network's gradient 1e-4 (FP32 activations, sums to 46 bits); the
diagnostics and statistics evaluate in FP64 from FP32 or FP64 fields; where two
calls run the same arithmetic, equality."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="no CUDA device")

from oracle import mlp_oracle as M  # noqa: E402
from oracle import oracle as O  # noqa: E402
from paper_2401_06841_gb300 import AdiabaticSolver, Solver  # noqa: E402
from paper_2401_06841_gb300 import inputs as I  # noqa: E402

TOL = {"f64": 1e-12, "f32": 1e-5}
DTYPE = {"f64": torch.float64, "f32": torch.float32}


def rel(got, ref):
    got = np.asarray(got, dtype=np.float64)
    return max(np.linalg.norm(got[:, v] - ref[:, v]) / max(np.linalg.norm(ref[:, v]), 1e-300)
               for v in range(ref.shape[1]))


def modes(kvec, seed):
    rng = np.random.default_rng(seed)
    kv = np.array(kvec, dtype=np.int32)
    return kv, rng.normal(size=(len(kv), 3, 2))


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("N,k,riemann", [(1, 1, "hll"), (2, 2, "hllc"), (3, 3, "rusanov"), (4, 1, "rusanov"),
                                         (7, 2, "hll"), (9, 3, "hllc"), (12, 1, "hllc"), (11, 2, "rusanov")])
def test_rhs_with_unaligned_result(N, k, riemann, prec):
    # driven and undriven; the result starts one element past a 16-byte boundary
    u = I.random_state(N, k, seed=500 + N)
    cfg = O.make_cfg(N, k, riemann=riemann)
    fo = O.Forcing(mach=2.0, zeta=0.5, seed=4)
    ahat = O.forcing_project(cfg, fo.kvec(), fo.amplitudes())
    dt = 0.3 * (1 / N) / ((k + 1) * 6.0)
    s = Solver(N, k, precision=prec, riemann=riemann)
    ud = torch.as_tensor(u, dtype=DTYPE[prec]).cuda()
    buf = torch.empty(ud.numel() + 1, dtype=DTYPE[prec], device="cuda")
    for a in (None, ahat):
        got = s.rhs(u, a, dt)
        assert rel(got.cpu().numpy(), O.rhs(cfg, u, a, dt)) < TOL[prec]
        ad = None if a is None else torch.as_tensor(a, dtype=DTYPE[prec]).cuda()
        torch.cuda.synchronize()
        rc = s.L.dg_rhs(s.h, ud.data_ptr(), None if ad is None else ad.data_ptr(), buf[1:].data_ptr(), dt)
        assert rc == 0
        assert torch.equal(buf[1:].view_as(got), got)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("N,k,riemann", [(4, 3, "hllc"), (7, 1, "rusanov"), (9, 2, "hllc"), (9, 2, "rusanov"),
                                         (6, 3, "rusanov"), (12, 1, "hllc")])
def test_adiabatic_rhs_with_unaligned_result(N, k, riemann, prec):
    u = I.random_energy_state(N, k, seed=600 + N, v_rms=0.3, p_mean=5.0, gamma=1.4)
    if prec == "f32":
        u = u.astype(np.float32).astype(np.float64)
    dt = 2e-3
    s = AdiabaticSolver(N, k, gamma=1.4, precision=prec, riemann=riemann)
    got = s.rhs(u, dt)
    ref = O.adi_rhs(O.make_cfg(N, k, riemann=riemann), 1.4, u, dt)
    # the momentum's condition number grows with the mesh: 3e-5 in FP32 as at 64^3
    assert rel(got.cpu().numpy(), ref) < (1e-12 if prec == "f64" else 3e-5)
    ud = torch.as_tensor(u, dtype=DTYPE[prec]).cuda()
    buf = torch.empty(ud.numel() + 1, dtype=DTYPE[prec], device="cuda")
    torch.cuda.synchronize()
    assert s.L.dg_adi_rhs(s.h, ud.data_ptr(), buf[1:].data_ptr(), dt) == 0
    assert torch.equal(buf[1:].view_as(got), got)


@pytest.mark.gpu
@pytest.mark.parametrize("N,k", [(1, 1), (3, 2), (5, 3), (65, 1), (66, 2)])
@pytest.mark.parametrize("kvec", [[(0, 0, 0)], [(-8, 8, -8), (8, -8, 8), (8, 8, 8)],
                                  [(1, 0, 0), (-1, 0, 0), (1, 0, 0), (0, -3, 2), (0, 3, -2), (-2, 5, 1), (2, 5, 1)]])
def test_forcing_modes_in_any_order_and_sign(N, k, kvec):
    # repeated modes, conjugate pairs, |k_d| = 8, rows of 64 cells and a remainder
    kv, amp = modes(kvec, 7)
    ref = O.forcing_project(O.make_cfg(N, k), kv, amp)
    # relative to the modes' size: on one cell most of them integrate to nothing
    scale = np.linalg.norm(ref) + 1e-3 * np.linalg.norm(amp)
    for prec in ("f64", "f32"):
        got = Solver(N, k, precision=prec).forcing_from_modes(kv, amp).cpu().numpy()
        assert np.linalg.norm(got - ref) < TOL[prec] * scale


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 4096])
def test_training_gradient_around_a_block_of_samples(k, n):
    D = 2 * I.nmodes(k)
    s = Solver(4, k, precision="f32", av="learned")
    th = M.init_params(D, seed=5).astype(np.float32)
    s.set_av_weights(th)
    rng = np.random.default_rng(n)
    X = rng.uniform(-1.5, 1.5, size=(n, D)).astype(np.float32)
    y = rng.normal(-2.0, 1.0, size=n).astype(np.float32)
    loss, g = s.mlp_grad(X, y)
    lref, gref = M.loss_and_grad(th.astype(np.float64), X.astype(np.float64), y.astype(np.float64))
    assert loss == pytest.approx(lref, rel=1e-5)
    assert np.linalg.norm(g.cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("N,k", [(1, 1), (1, 2), (3, 2), (6, 2), (4, 3)])
def test_statistics_and_diagnostics_on_small_grids(N, k, prec):
    # grids of 2, 3, 9, 18 and 16 points; one cell with exact zeros (its rows take the
    # conversion instruction)
    u = I.random_state(N, k, seed=700 + N, v_rms=0.8)
    u[0, 1:, :] = 0.0
    if prec == "f32":
        u = u.astype(np.float32).astype(np.float64)
    cfg = O.make_cfg(N, k)
    s = Solver(N, k, precision=prec)
    s.set_state(u)
    assert np.abs(s.density_pdf(-1.0, 1.0, 37) - O.density_pdf(cfg, u, -1.0, 1.0, 37)).max() < 1e-13
    l, v = s.structure_function(nbins=5, npairs=333, seed=9)
    lr, vr = O.structure_function(cfg, u, 5, 333, 9)
    assert np.allclose(l, lr, rtol=1e-14, atol=0) and np.allclose(v, vr, rtol=1e-11, atol=0)
    km, pw, cnt = s.power_spectrum(11)
    kr, pr, cr = O.power_spectrum(cfg, u, 11)
    assert np.array_equal(cnt, cr)
    assert np.allclose(km, kr, rtol=1e-13, atol=0)
    assert np.allclose(pw, pr, rtol=1e-10, atol=1e-18 * max(pr.max(), 1.0))
    got, ref = s.diagnostics(1e-3), O.diagnostics(cfg, u, None, 1e-3)
    tol = 1e-12 if prec == "f64" else 2e-5
    for key in ("mass", "mom_x", "mom_y", "mom_z", "ekin", "mach", "mach_rho", "rho_min", "rho_max", "max_speed",
                "av_work"):
        assert got[key] == pytest.approx(ref[key], rel=tol, abs=tol * 10), key
    assert got["av_frac"] == pytest.approx(ref["av_frac"], abs=0.02 if prec == "f32" else 1e-12)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,N,k,mach,kw", [
    ("iso", 5, 1, 3.0, dict(precision="f64")), ("iso", 6, 2, 1.0, dict(precision="f32")),
    ("iso", 5, 3, 2.0, dict(precision="f32", positivity="repeat")), ("iso", 5, 3, 3.0, dict(precision="f32", av="learned")),
    ("iso", 5, 3, 1.0, dict(precision="f32", av="learned", fused_infer=True)), ("adi", 5, 2, 2.0, dict(precision="f32")),
    ("adi", 6, 1, 2.0, dict(precision="f64"))])
def test_driven_steps_in_one_call_and_one_by_one(kind, N, k, mach, kw):
    # driving updated at some steps or at all: nine steps at once, one at a time, and
    # four, then a resumed context for five, are the same bit for bit, with the same
    # random numbers left
    def make():
        if kind == "iso":
            s = Solver(N, k, **kw)
            if kw.get("av") == "learned":
                s.set_av_weights(M.init_params(2 * I.nmodes(k), seed=5).astype(np.float32))
            s.set_state(I.random_state(N, k, seed=800, v_rms=0.3))
            s.set_forcing(mach=mach, zeta=0.5, seed=3)
        else:
            s = AdiabaticSolver(N, k, gamma=1.4, **kw)
            s.set_state(I.random_energy_state(N, k, seed=800, v_rms=0.3, p_mean=5.0, gamma=1.4))
            s.set_forcing(mach=mach, zeta=0.5, seed=3, cs_ref=1.0)
        return s

    def end(s):
        m = s.get_meta()
        return s.get_state(), bytes(C.string_at(C.addressof(m), C.sizeof(m)))

    a, b, c = make(), make(), make()
    a.step(9)
    for _ in range(9):
        b.step(1)
    c.step(4)
    u, m = c.get_state(), c.get_meta()
    d = make()
    d.set_state(u)
    d.set_meta(m)
    d.step(5)
    ua, ma = end(a)
    for s in (b, d):
        us, ms = end(s)
        assert torch.equal(us, ua)
        assert ms == ma
