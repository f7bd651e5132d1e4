"""lb_moments without sums (pairs of nodes over all nodes, solid ones
included) against the oracle and against the same call with sums, for pairs
that straddle rows and walls, odd node counts and outputs off pair alignment."""
import numpy as np
import pytest

from parity_util import check

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402


@pytest.mark.gpu
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("walls,shape", [(False, (1, 1, 1)), (False, (3, 1, 1)), (False, (8, 3, 5)), (False, (7, 5, 3)), (True, (1, 1, 3)),
                                         (True, (3, 3, 4)), (True, (6, 5, 3)), (True, (65, 3, 5)), (True, (130, 2, 3))])
def test_fields(ora, walls, shape, shift):
    n = shape[0] * shape[1] * shape[2]
    u = inputs.gaussian_field(shape, 3, 5e-3, seed=1)
    rho = 1.0 + inputs.gaussian_field(shape, 1, 5e-3, seed=2)[0]
    f = inputs.gaussian_field(shape, 3, 1e-4, seed=3).astype(np.float32)
    bf = (1e-5, -2e-5, 3e-6)
    p = ora.make_params(shape, walls=walls, body_force=bf)
    pops = ora.step(p, ora.equilibrium(p, rho, u), f.astype(np.float64), 0)
    lat = L.Lattice(shape, walls=walls, body_force=bf, force=torch.as_tensor(f).cuda())
    lat.set_populations(torch.as_tensor(pops).cuda())
    out = [torch.full((c * n + 4,), np.nan, dtype=torch.float32, device="cuda")[shift:shift + c * n] for c in (1, 3, 6)]
    L.lb_moments(lat.h, *out)
    got = [x.cpu().numpy().astype(np.float64).reshape((-1,) + shape[::-1]) for x in out]
    want = ora.moments(p, pops, f.astype(np.float64))
    fl = slice(1, -1) if walls else slice(None)
    for nm, x, y, base in zip(("rho", "j", "pi"), got, want, (1.0, 0.0, 0.0)):
        # FP32 sums of 19 deviations of order 5e-3 on fields of order one (j: 5e-3)
        check("%s %s" % (nm, shape), x[:, fl], np.reshape(y, x.shape)[:, fl], 2e-6, 5e-6)
        if walls:
            for z in (0, -1):
                assert (x[:, z] == base).all()
    with_sums = [torch.empty_like(x) for x in out]
    L.lb_moments(lat.h, *with_sums, torch.empty(L.LB_NSUMS, dtype=torch.float64, device="cuda"))
    for x, y in zip(out, with_sums):
        assert torch.allclose(x, y, rtol=1e-6, atol=1e-8)
    lat.close()
