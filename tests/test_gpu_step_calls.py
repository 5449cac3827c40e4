"""Steps in one call and one by one where the driving's next update is foreseen
wrongly or a step is repeated.  Within a call dg_step leaves out the projection at the
end of a step when the next one is expected to start with an update of the driving
(by the previous dt); the last step of a call never does.  Whatever was foreseen,
the states, times and random numbers are the same bit for bit.  And x3 by default
is the FP32 arithmetic."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="no CUDA device")

from paper_2401_06841_gb300 import Solver  # noqa: E402
from paper_2401_06841_gb300 import inputs as I  # noqa: E402


def same(a, b):
    ma, mb = a.get_meta(), b.get_meta()
    return torch.equal(a.get_state(), b.get_state()) and \
        C.string_at(C.addressof(ma), C.sizeof(ma)) == C.string_at(C.addressof(mb), C.sizeof(mb))


@pytest.mark.gpu
@pytest.mark.parametrize("k,prec", [(1, "f64"), (2, "f32"), (3, "f32")])
def test_driving_update_foreseen_but_not_due(k, prec):
    # updates every 1/(200 mach) = 0.01: after three steps of 0.003 the next is expected
    # at t = 0.012, but the steps go on with 0.0002
    def make():
        s = Solver(5, k, precision=prec)
        s.set_state(I.random_state(5, k, seed=810, v_rms=0.3))
        s.set_forcing(mach=0.5, zeta=0.5, seed=3)
        s.step(3, fixed_dt=0.003)
        return s

    a, b = make(), make()
    a.profile(True)
    assert a.step(3, fixed_dt=0.0002)[0] == pytest.approx(0.0096, rel=1e-12)
    for _ in range(3):
        b.step(1, fixed_dt=0.0002)
    # one projection per step, the state's own carried over from the steps before
    assert a.profile_read()["n_project"] == 3
    assert same(a, b)
    assert a.step(2, fixed_dt=0.0003) == (b.step(1, fixed_dt=0.0003), b.step(1, fixed_dt=0.0003))[1]
    assert same(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_repeated_step_before_a_driving_update(prec):
    # two streams part at x = 1/2 with 3 cs: the cell beside the plane loses 12 dt of its
    # mass in a stage, so a step of 0.1 fails in its first stage and is repeated with
    # half the dt or less.  Updates every 0.001 are foreseen for every step but the
    # call's last
    N, k = 4, 1
    u = np.zeros((N ** 3, 4, I.nmodes(k)))
    u[:, 0, 0] = 1.0
    u[:, 1, 0] = np.where(np.arange(N ** 3) % N < N // 2, -3.0, 3.0)

    def make():
        s = Solver(N, k, precision=prec)
        s.set_state(u)
        s.set_forcing(mach=5.0, zeta=0.5, seed=3)
        s.step(1, fixed_dt=0.0006)
        return s

    a, b = make(), make()
    assert b.step(1, fixed_dt=0.1)[1] in (0.05, 0.025, 0.0125)
    for _ in range(2):
        b.step(1, fixed_dt=0.001)
    a.step(1, fixed_dt=0.1)
    c = make()
    c.step(2, fixed_dt=0.1)
    d = make()
    for _ in range(2):
        d.step(1, fixed_dt=0.1)
    assert same(c, d)
    a.step(2, fixed_dt=0.001)
    assert same(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 2, 3])
def test_x3_by_default_is_fp32(k):
    N = 5
    u = I.random_state(N, k, seed=820 + k, v_rms=0.5)
    out = {}
    for prec in ("f32", "x3"):
        s = Solver(N, k, precision=prec)
        s.set_state(u)
        s.set_forcing(mach=2.0, zeta=0.5, seed=3)
        s.step(3)
        out[prec] = (s, s.rhs(u, s.ahat.clone(), 1e-3), s.project_velocity(u))
    assert same(out["f32"][0], out["x3"][0])
    assert all(torch.equal(p, q) for p, q in zip(out["f32"][1:], out["x3"][1:]))
