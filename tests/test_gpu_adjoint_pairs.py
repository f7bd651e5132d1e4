"""The reverse step's pairs of nodes where they straddle rows, planes and
walls, and caller buffers that start at any element: one step against the
oracle, and against the same call on aligned buffers."""
import numpy as np
import pytest

from parity_util import check

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu
GAM = dict(gamma_shear=0.2, gamma_bulk=-0.3, gamma_odd=0.4, gamma_even=-0.1)


def _lambda(lat, lam, shift):
    pitch = L.lb_plane_pitch(lat.params)
    t = torch.zeros(19 * pitch + 4, dtype=torch.float32, device="cuda")[shift:shift + 19 * pitch].view(19, pitch)
    if lam is not None:
        t[:, :lat.n_nodes] = torch.as_tensor(lam.reshape(19, -1).astype(np.float32)).cuda()
    return t


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("walls,shape", [(False, s) for s in [(1, 1, 1), (2, 1, 3), (3, 3, 3), (8, 5, 6), (65, 3, 4), (130, 2, 3)]] +
                         [(True, s) for s in [(1, 1, 3), (2, 1, 3), (3, 3, 4), (8, 5, 6), (65, 3, 5), (130, 2, 4)]])
def test_one_step(ora, walls, shape, shift):
    bf = (2e-4, -1e-4, 0.0 if walls else 1e-4)
    u = inputs.gaussian_field(shape, 3, 5e-3, seed=1)
    f = inputs.gaussian_field(shape, 3, 1e-3, seed=2).astype(np.float32)
    lam = inputs.gaussian_field(shape, 19, 1.0, seed=3).astype(np.float32).astype(np.float64)
    if walls:
        for x in (u, f, lam):
            x[:, 0] = x[:, -1] = 0
    p = ora.make_params(shape, walls=walls, body_force=bf, **GAM)
    s0 = ora.equilibrium(p, None, u)
    want, want_g = ora.adjoint_step(p, s0, lam, f.astype(np.float64))
    lat = L.Lattice(shape, walls=walls, body_force=bf, force=torch.as_tensor(f).cuda(), **GAM)
    lat.set_populations(torch.as_tensor(s0).cuda())
    cur, _ = L.lb_state_buffers(lat.h)
    out = _lambda(lat, None, shift)
    g = torch.zeros((3,) + shape[::-1], dtype=torch.float32, device="cuda")
    L.lb_adjoint_step(lat.h, cur, _lambda(lat, lam, shift), out, g)
    got = out[:, :lat.n_nodes].double().cpu().numpy().reshape((19,) + shape[::-1])
    fl = slice(1, -1) if walls else slice(None)
    # the bars of the single-step comparison on larger boxes: FP32 sums of 19 terms
    check("adjoint pair %s lambda" % (shape,), got[:, fl], want[:, fl], 1e-5, 5e-5)
    check("adjoint pair %s gradient" % (shape,), g.cpu().numpy()[:, fl], want_g[:, fl], 1e-5, 5e-5)
    if walls:
        assert not got[:, 0].any() and not got[:, -1].any()  # solid entries stay zero
    lat.close()


@pytest.mark.parametrize("dtype", [L.LB_F32, L.LB_F16])
@pytest.mark.parametrize("shape", [(6, 5, 4), (7, 5, 4), (512, 2, 2)])
def test_step_from_unaligned(shape, dtype):
    """lb_step_from on buffers that start one element after a pair boundary."""
    lat = L.Lattice(shape, kT=1e-4, seed=3, dtype=dtype)
    lat.init_equilibrium(None, torch.as_tensor(inputs.gaussian_field(shape, 3, 5e-3, seed=1)).cuda())
    kind = torch.float32 if dtype == L.LB_F32 else torch.float16
    n = lat._bufs[0].numel() // kind.itemsize
    src = lat._bufs[0].view(kind)
    want = torch.zeros(n, dtype=kind, device="cuda")
    L.lb_step_from(lat.h, src, want, 4)
    a, b = (torch.zeros(n + 8, dtype=kind, device="cuda")[1:n + 1] for _ in range(2))
    a.copy_(src)
    L.lb_step_from(lat.h, a, b, 4)
    nodes, pitch = lat.n_nodes, n // 19
    assert torch.equal(b.view(19, pitch)[:, :nodes], want.view(19, pitch)[:, :nodes])
    lat.sync()
    lat.close()
