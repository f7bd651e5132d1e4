"""The linear mapping of the stream-collide launch (two consecutive nodes a
thread over the fluid's index range) where its pairs straddle rows, planes and
the walls, and where an odd number of nodes leaves a lone one: one step from a
perturbed state against the oracle, in every storage format."""
import numpy as np
import pytest

from parity_util import check

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu

PERIODIC = [(1, 1, 1), (1, 1, 2), (1, 2, 1), (3, 1, 1), (2, 1, 3), (3, 3, 3), (5, 3, 4), (63, 2, 1), (65, 3, 5), (129, 1, 3),
            (30, 7, 5), (254, 3, 2), (258, 2, 3)]
WALLS = [(1, 1, 3), (1, 3, 4), (2, 1, 3), (3, 1, 3), (3, 3, 5), (5, 5, 3), (4, 3, 3), (65, 3, 4), (63, 5, 5), (130, 3, 4)]
# one step: FP32 arithmetic; FP16 / BF16: two roundings to 11 / 8 bits
BARS = {L.LB_F32: (2e-6, 5e-6), L.LB_F16: (2.0 ** -10, 2.0 ** -10), L.LB_BF16: (2.0 ** -7, 2.0 ** -7)}


@pytest.mark.parametrize("dtype", sorted(BARS))
@pytest.mark.parametrize("kT", [0.0, 1e-4])
@pytest.mark.parametrize("walls,shape", [(False, s) for s in PERIODIC] + [(True, s) for s in WALLS])
def test_one_step(ora, walls, shape, kT, dtype):
    u = inputs.shear_wave(shape, 0.02) + inputs.gaussian_field(shape, 3, 5e-3, seed=1)
    rho = 1.0 + inputs.gaussian_field(shape, 1, 5e-3, seed=2)[0]
    field = inputs.gaussian_field(shape, 3, 1e-4, seed=3).astype(np.float32)
    kw = dict(kT=kT, seed=5, walls=walls, body_force=(1e-5, -2e-5, 3e-6), gamma_shear=0.2, gamma_odd=0.4)
    p = ora.make_params(shape, **kw)
    start = ora.equilibrium(p, rho, u)
    want = ora.step(p, start, field.astype(np.float64), 0)
    lat = L.Lattice(shape, dtype=dtype, force=torch.as_tensor(field).cuda(), **kw)
    lat.init_equilibrium(torch.as_tensor(rho).cuda(), torch.as_tensor(u).cuda())
    lat.step(1)
    got = lat.get_populations().cpu().numpy()
    fluid = slice(1, -1) if walls else slice(None)
    a = ora.tables()[1][:, None, None, None]
    check("linear %s" % (shape,), (got - a)[:, fluid], (want - a)[:, fluid], *BARS[dtype])
    lat.close()
