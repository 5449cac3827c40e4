"""The density PDF and the spectrum on both sides of the rule that gives a thread a
row of points (below 64 cells per multiprocessor) or a whole cell, with fewer and
more bins than a block has samples (counters of the block's own or the common ones).
FP64 from the same FP32-representable coefficients as the oracle.  Bounds: the
histogram's counts are integers here, while the oracle adds its n = N^3 (k+1)^3 weights one
by one, each addition rounding by at most 2^-53 of the sum: 1e-13 + n 2^-53 h, and so for
the |kappa| of a shell's modes; a shell's power 1e-10 as in test_gpu_shapes.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="no CUDA device")

from oracle import oracle as O  # noqa: E402
from paper_2401_06841_gb300 import Solver  # noqa: E402
from paper_2401_06841_gb300 import inputs as I  # noqa: E402


def edge():
    """the largest mesh taken by rows and the smallest by cells"""
    n = 1
    while (n + 1) ** 3 < 64 * torch.cuda.get_device_properties(0).multi_processor_count:
        n += 1
    return n, n + 1


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("side", [0, 1])
def test_pdf_and_spectrum_by_rows_and_by_cells(side, k, prec):
    N = edge()[side]
    u = I.random_state(N, k, seed=850 + k, v_rms=0.8).astype(np.float32).astype(np.float64)
    cfg = O.make_cfg(N, k)
    s = Solver(N, k, precision=prec)
    s.set_state(u)
    for nbins in (1, 37, 129, 1025, 2000):
        h = s.density_pdf(-0.5, 0.5, nbins)
        ref = O.density_pdf(cfg, u, -0.5, 0.5, nbins)
        assert (np.abs(h - ref) <= 1e-13 + N ** 3 * (k + 1) ** 3 * 2.0 ** -53 * ref).all()
        assert np.array_equal(h, s.density_pdf(-0.5, 0.5, nbins))  # integer counts: the same bits
    km, pw, cnt = s.power_spectrum(23)
    kr, pr, cr = O.power_spectrum(cfg, u, 23)
    assert np.array_equal(cnt, cr)
    assert (np.abs(km - kr) <= (1e-13 + cr * 2.0 ** -53) * kr).all()
    assert np.allclose(pw, pr, rtol=1e-10, atol=1e-18 * max(pr.max(), 1.0))
