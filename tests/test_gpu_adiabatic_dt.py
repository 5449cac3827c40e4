"""The adiabatic CFL step in FP32 takes correctly rounded sound speeds: a uniform gas
at rest has dt = cfl h / ((k+1) 3 c) with c = sqrt(gamma p / rho), where every operation
on the device is one rounding of single precision, so that numpy's float32 gives the
same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="no CUDA device")

from paper_2401_06841_gb300 import AdiabaticSolver  # noqa: E402
from paper_2401_06841_gb300 import inputs as I  # noqa: E402


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 2, 3])
def test_sound_speed_of_a_uniform_gas(k):
    N, gamma, cfl = 2, 1.4, 0.3
    f = np.float32
    s = AdiabaticSolver(N, k, gamma=gamma, precision="f32", cfl=cfl)
    u = np.zeros((N ** 3, 5, I.nmodes(k)), dtype=f)
    u[:, 0, 0] = 1.0
    for e in np.random.default_rng(4).uniform(0.5, 40.0, 64).astype(f):
        u[:, 4, 0] = e
        s.set_state(u)
        p = f(gamma - 1.0) * e
        smax = f(3.0) * np.sqrt(f(gamma) * p)
        # (the quotient in FP64: an ulp of smax is 6e-8 or more of it)
        assert s.step(1)[1] == pytest.approx(cfl / N / (k + 1) / float(smax), rel=1e-14), float(e)
