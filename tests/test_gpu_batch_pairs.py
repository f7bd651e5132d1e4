"""Batched replicas whose pairs of nodes straddle rows and planes or end
alone, in tiles that do not fill a block or have an odd length, against the
oracle; with and without forces, and with the mode records."""
import numpy as np
import pytest

from parity_util import check

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu
SHAPES = [(1, 1, 1), (3, 1, 1), (1, 1, 5), (3, 3, 3), (5, 3, 4), (7, 5, 9), (8, 6, 5), (33, 4, 3), (64, 3, 2)]


@pytest.mark.parametrize("dtype,bars", [(L.LB_F32, (2e-6, 5e-6)), (L.LB_F16, (2.0 ** -9, 2.0 ** -9))])
@pytest.mark.parametrize("tile", [32, 33, 2048])
@pytest.mark.parametrize("force,records", [((0.0, 0.0, 0.0), False), ((1e-4, -2e-4, 5e-5), True)])
def test_uneven_replicas(ora, dtype, bars, tile, force, records):
    n, steps = len(SHAPES), 2
    kw = dict(kT=1e-4, body_force=force, gamma_shear=0.2, gamma_bulk=-0.1, gamma_even=0.05)
    stream = torch.cuda.Stream()
    B = L.Batch(SHAPES, seeds=[21 + k for k in range(n)], dtype=dtype, stream=stream, **kw)
    L.lb_batch_set_config(B.b, 64, tile, 2)
    us = [inputs.gaussian_field(s, 3, 1e-2, seed=30 + k) for k, s in enumerate(SHAPES)]
    rec = torch.empty((n, steps, 12), dtype=torch.float64, device="cuda")
    with torch.cuda.stream(stream):
        for k, u in enumerate(us):
            L.lb_batch_init_equilibrium(B.b, k, None, torch.as_tensor(u).cuda())
        torch.cuda.synchronize()
        if records:
            L.lb_batch_record_modes(B.b, rec, steps)
        L.lb_batch_step(B.b, steps, False)
    L.lb_batch_sync(B.b)
    a = ora.tables()[1][:, None, None, None]
    for k, s in enumerate(SHAPES):
        p = ora.make_params(s, seed=21 + k, replica=k, **kw)
        state = ora.equilibrium(p, None, us[k])
        for t in range(steps):
            if records and dtype == L.LB_F32:
                rho, j, _ = ora.moments(p, state, None)
                u = j / rho
                ph = [np.exp(-2j * np.pi * np.arange(m) / m) for m in s]
                want = [(u[0] * ph[2][:, None, None]).sum(), (u[1] * ph[2][:, None, None]).sum(), (u[1] * ph[0]).sum(),
                        (u[2] * ph[0]).sum(), (u[2] * ph[1][:, None]).sum(), (u[0] * ph[1][:, None]).sum()]
                got = rec[k, t].cpu().numpy()
                w = np.array([[v.real, v.imag] for v in want]).ravel()
                # FP32 sums of up to 384 velocities of order 1e-2
                assert np.abs(got - w).max() < 2e-6 * np.abs(u).sum() / 3 + 1e-9
            state = ora.step(p, state, None, t)
        got = B.get_populations(k).cpu().numpy()
        check("batch %s" % (s,), got - a, state - a, *bars)
    B.close()
