"""The count of gated tiles (dg_prof): tiles whose div v was skipped, not tiles
whose coefficients are zero.  A network that reads the cells' speed alone and a
gate between rest and motion fix which coefficients are zero; the volume kernel
skips the 32 consecutive cells of a block together."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="no CUDA device")

from paper_2401_06841_gb300 import Solver  # noqa: E402
from paper_2401_06841_gb300 import inputs as I  # noqa: E402


def weights(k):
    # y = gelu(gelu(|v|_0 / cs)): 0 at rest, 1.9 at 2 cs
    D, H = 2 * I.nmodes(k), 64
    w1, b1, w2, b2, w3, b3 = np.zeros((H, D)), np.zeros(H), np.zeros((H, H)), np.zeros(H), np.zeros(H), np.zeros(1)
    w1[0, D // 2] = w2[0, 0] = w3[0] = 1.0
    return np.concatenate([w1.ravel(), b1, w2.ravel(), b2, w3, b3]).astype(np.float32)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("moving,blocks", [([], 0), ([20], 1), ([5, 63], 2), ([15, 16], 1)])
def test_a_tile_beside_an_active_one_of_its_block_is_not_gated(moving, blocks, k, prec):
    N, tile = 4, 32 if k == 1 else 16  # two blocks of 32 cells
    u = np.zeros((N ** 3, 4, I.nmodes(k)))
    u[:, 0, 0] = 1.0
    u[moving, 1, 0] = 2.0
    s = Solver(N, k, precision=prec, av="learned", nu_gate=2.0)
    s.set_av_weights(weights(k))
    s.set_state(u)
    nu = s.av_nu().cpu().numpy()
    assert sorted(np.flatnonzero(nu)) == moving
    s.profile(True)
    s.rhs(u, None, 1e-3)
    p = s.profile_read()
    assert p["tiles_volume"] == 64 // tile
    assert p["tiles_gated"] == (2 - blocks) * 32 // tile
