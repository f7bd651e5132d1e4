"""The relaxation keeps a second moment that is at its equilibrium: the
rounding of its constants is no factor on it.  A nearly uniform flow, one step
against the oracle's step of the same stored state, and of the error of each
second moment the part that is proportional to the moment, for eigenvalues
whose multiples round badly against a neighbour whose multiples are exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu
EXACT = -199.0 / 256.0  # gamma / w, (1 - gamma) / w, gamma - 1 and 1 + gamma are FP32 values


def _gains(ora, gamma, shape, forced):
    x, y, z = (2 * np.pi * np.arange(m) / m for m in shape)
    u = np.empty((3,) + shape[::-1])
    u[0] = 0.15 + 0.03 * np.sin(z)[:, None, None]
    u[1] = 0.15 + 0.03 * np.sin(x)[None, None, :]
    u[2] = 0.15 + 0.03 * np.sin(y)[None, :, None]
    kw = dict(kT=0.0, gamma_shear=gamma, gamma_bulk=gamma, body_force=(1e-4, -2e-4, 1e-4) if forced else (0.0, 0.0, 0.0))
    lat = L.Lattice(shape, **kw)
    lat.init_equilibrium(None, torch.as_tensor(u).cuda())
    start = lat.get_populations().cpu().numpy()
    lat.step(1)
    got = lat.get_populations().cpu().numpy()
    lat.close()
    want = ora.step(ora.make_params(shape, **kw), start, None, 0)
    c, a, e, w, opp = ora.tables()
    out = {}
    for k in range(4, 10):
        m = np.tensordot(e[k], want - a[:, None, None, None], axes=1)
        err = np.tensordot(e[k], got - want, axes=1)
        if np.sqrt((m * m).mean()) >= 5e-3:  # (modes 5 and 6 may nearly vanish: all components are alike)
            out[k] = (err * m).sum() / (m * m).sum()
    return out


# gamma / w and (1 - gamma) / w, each rounded to FP32, miss 1 / w by 1.06e-7 (w = 1/9), one up and one down
@pytest.mark.parametrize("gamma", [-0.7779287695884705, -0.7779934406280518])
@pytest.mark.parametrize("shape", [(48, 48, 48), (47, 48, 49), (256, 24, 16)])
@pytest.mark.parametrize("forced", [False, True])
def test_no_gain(ora, gamma, shape, forced):
    got, ref = _gains(ora, gamma, shape, forced), _gains(ora, EXACT, shape, forced)
    for k in got:
        # a node's second moment carries some 4e-9 of rounding (twelve stored values below 2^-5) against 2e-2:
        # the projection averages it over 1e5 nodes to 1e-9 at most.  What else is proportional to the moment
        # (the FP32 weights, a constant force added to values on a grid) is that of the neighbour to 1e-3.
        assert abs(got[k] - ref[k]) < 1e-8, (k, got[k], ref[k])
