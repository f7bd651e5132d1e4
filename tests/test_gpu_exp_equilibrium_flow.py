"""The exponential equilibrium on both sides of |u| = 0.1, where the update
goes from one Newton step with the Jacobian of rest to two full ones, on rows
of even and odd length and between walls: one step against the oracle."""
import numpy as np
import pytest

from parity_util import check

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402


@pytest.mark.gpu
@pytest.mark.parametrize("speed", [1e-4, 0.05, 0.0999, 0.1001, 0.15, 0.25])
@pytest.mark.parametrize("walls,shape", [(False, (8, 6, 5)), (False, (7, 5, 9)), (False, (1, 1, 5)), (True, (6, 5, 5)),
                                         (True, (5, 5, 4)), (False, (130, 3, 2))])
def test_one_step(ora, walls, shape, speed):
    d = inputs.gaussian_field(shape, 3, 1.0, seed=7)
    u = speed * d / np.sqrt((d * d).sum(0))  # every direction, the speed exactly
    if walls:
        u[:, 0] = u[:, -1] = 0
    kw = dict(gamma_shear=0.3, gamma_bulk=-0.2, gamma_odd=0.4, gamma_even=-0.1, walls=walls, equilibrium=1)
    p = ora.make_params(shape, **kw)
    # start from rest and give the nodes their velocity by the force: f / 2 = rho u
    f = (2.0 * u).astype(np.float32)
    rest = ora.equilibrium(p, None, None)
    want = ora.step(p, rest, f.astype(np.float64), 0)
    lat = L.Lattice(shape, force=torch.as_tensor(f).cuda(), **kw)
    lat.init_equilibrium()
    lat.step(1)
    got = lat.get_populations().cpu().numpy()
    fl = slice(1, -1) if walls else slice(None)
    a = ora.tables()[1][:, None, None, None]
    # FP32 rounding of a one-step comparison, as for the quadratic equilibrium
    check("exp %s u %g" % (shape, speed), (got - a)[:, fl], (want - a)[:, fl], 2e-6, 5e-6)
    lat.close()
