"""Face fluxes where the flow crosses the whole wave fan: HLL and HLLC return the
flux of the upwind side alone, in both directions alike, however dense the other
side is.  Cells of constant density and velocity, a dense half of the mesh
(1e6) beside a thin one (1), the flow along an axis at 1.5 to 10 cs with another
speed in every column, tangential velocities that differ between the halves.

The thin cells whose upwind neighbour is thin hold nothing of the dense half in
their right-hand side: it is compared with the FP64 oracle cell by cell, relative to
the thin gas's own flux rho (|v| + cs)^2 / h.  Bounds as for one evaluation in
test_gpu_parity.py: FP64 1e-12, FP32 1e-5 (a flux is some twenty operations, a
cell's right-hand side the sum of six and the volume term)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="no CUDA device")

from oracle import oracle as O  # noqa: E402
from paper_2401_06841_gb300 import Solver  # noqa: E402
from paper_2401_06841_gb300 import inputs as I  # noqa: E402

N, DENSE = 8, 1e6
TOL = {"f64": 1e-12, "f32": 1e-5}


def state(k, axis, sign, seed):
    """Coefficients [N^3, 4, b] in FP32-representable numbers, and the thin cells
    past the first from the dense half (numbered against the flow)."""
    rng = np.random.default_rng(seed)
    pos = np.indices((N, N, N))[2 - axis]  # arrays are [z, y, x]
    thin = pos >= N // 2
    rho = np.where(thin, 1.0, DENSE)
    vn = np.expand_dims(rng.uniform(1.5, 10.0, size=(N, N)), 2 - axis) * np.ones((N, N, N))
    v = np.where(thin[None], 0.7, -1.3) * np.ones((3, N, N, N))
    v[axis] = sign * vn
    u = np.zeros((N ** 3, 4, I.nmodes(k)))
    u[:, 0, 0] = rho.ravel()
    for d in range(3):
        u[:, 1 + d, 0] = (rho * v[d]).ravel()
    # left-going flow enters the thin half through its upper boundary, from the dense half
    inner = thin & (pos != (N - 1 if sign < 0 else N // 2))
    scale = ((np.abs(v).sum(0) + 1.0) ** 2 * N).ravel()
    return u.astype(np.float32).astype(np.float64), inner.ravel(), scale


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("riemann", ["hll", "hllc"])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_upwind_flux_of_a_thin_gas_beside_a_dense_one(k, riemann, prec):
    s = Solver(N, k, precision=prec, riemann=riemann, av="off")
    cfg = O.make_cfg(N, k, av_mode=0, riemann=riemann)
    for axis in range(3):
        for sign in (-1.0, 1.0):
            u, inner, scale = state(k, axis, sign, seed=90 + axis)
            got = s.rhs(u, None, 0.0).cpu().numpy().astype(np.float64)
            err = np.abs(got - O.rhs(cfg, u, None, 0.0))[inner].max(axis=(1, 2)) / scale[inner]
            assert err.max() < TOL[prec], (axis, sign, err.max())


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("riemann", ["hll", "hllc"])
@pytest.mark.parametrize("bad", ["nan", "vacuum"])
def test_a_downwind_vacuum_or_nan_does_not_enter(bad, riemann, prec):
    # uniform flow at 3 cs along an axis past one cell of NaN or of nothing (its velocity is
    # 0/0): the cell upwind of it has the right-hand side of the undisturbed flow
    k, n = 2, 8
    s = Solver(n, k, precision=prec, riemann=riemann, av="off")
    for axis in range(3):
        for sign in (-1, 1):
            u = I.random_state(n, k, seed=95, v_rms=0.1)
            u[:, 1 + axis] += 3.0 * sign * u[:, 0]
            c = (3 * n + 4) * n + 5
            up = c - sign * (1, n, n * n)[axis]
            ref = s.rhs(u, None, 0.0)
            u[c] = np.nan if bad == "nan" else 0.0
            got = s.rhs(u, None, 0.0)
            assert torch.equal(got[up], ref[up]), (axis, sign)
