"""The re-update of impulse nodes after an overlapped coupling in 16-bit
storage: it reads a node's impulse and then clears it, and the cleared value
must not be what the update sees."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu


def _run(shape, dtype, overlap, kernel, kT=0.0, seed=3, steps=1, walls=False, pos0=(5.3, 6.6, 4.2)):
    lat = L.Lattice(shape, kT=kT, seed=seed, dtype=dtype, walls=walls)
    lat.init_equilibrium()
    pos = torch.tensor([pos0], dtype=torch.float64).cuda()
    mom = torch.tensor([[0.06, -0.04, 0.03]], dtype=torch.float32).cuda()
    parts = L.particles(1, pos, mom, gamma0=2.0)
    out = []
    for t in range(steps):
        cp = L.couple_params(n_substeps=4, dt=0.1, seed=5, md_step0=4 * t, kernel=kernel, overlap=overlap)
        L.lb_couple_particles(lat.h, parts, cp)
        lat.step(1)
        out.append(lat.get_populations().cpu().numpy())
    lat.step(1)  # nothing is left to be applied again
    out.append(lat.get_populations().cpu().numpy())
    assert lat.sync()[1] == 0
    lat.close()
    return out


@pytest.mark.parametrize("dtype,mantissa", [(L.LB_F16, 10), (L.LB_BF16, 7)])
@pytest.mark.parametrize("kernel", [2, 3, 4])
def test_impulse_is_applied_once(ora, dtype, mantissa, kernel):
    shape = (12, 13, 11)
    a = ora.tables()[1][:, None, None, None]
    got, want = _run(shape, dtype, True, kernel), _run(shape, dtype, False, kernel)
    for t, (x, y) in enumerate(zip(got, want)):
        x, y = x - a, y - a
        assert np.abs(y).max() > 1e-4  # the particle moved the fluid
        # each update stores within half a unit in the last place of the same FP32 value, so the two
        # orders are a unit apart at most, and a second update carries the unit of the first
        assert np.abs(x - y).max() <= (t + 1) * 2.0 ** -mantissa * np.abs(y).max()


@pytest.mark.parametrize("dtype", [L.LB_F16, L.LB_BF16])
@pytest.mark.parametrize("kernel", [2, 4])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("eigenvalues", [{}, {"gamma_shear": 0.2, "gamma_bulk": -0.1, "gamma_odd": 0.1, "gamma_even": 0.05}])
def test_rounds_as_the_packed_update(dtype, kernel, walls, eigenvalues):
    """A node updated again by itself gives the bits that the update of all
    nodes gives for the same impulses (with noise): particles eight nodes apart,
    whose stencils do not meet, so that the impulse sums are the same too."""
    shape = (64, 56, 48)
    grid = np.stack(np.meshgrid(*[np.arange(4, s - 4, 8) for s in shape], indexing="ij"), -1).reshape(-1, 3)
    pos0 = grid + np.random.default_rng(1).uniform(0, 1, grid.shape)
    field = torch.as_tensor(inputs.gaussian_field(shape, 3, 1e-5, seed=3), dtype=torch.float32).cuda() if walls else None
    u = torch.as_tensor(inputs.gaussian_field(shape, 3, 1e-2, seed=4)).cuda()
    out = []
    for overlap in (False, True):
        lat = L.Lattice(shape, kT=1e-4, seed=3, dtype=dtype, walls=walls, force=field, **eigenvalues)
        lat.init_equilibrium(None, u)
        n = len(pos0)
        mom = torch.as_tensor(inputs.maxwell_momenta(n, 1.0, 1e-4, seed=2), dtype=torch.float32).cuda()
        parts = L.particles(n, torch.as_tensor(pos0).cuda(), mom, gamma0=2.0)
        L.lb_couple_particles(lat.h, parts, L.couple_params(n_substeps=3, dt=0.1, seed=5, kernel=kernel, overlap=overlap))
        lat.step(1)
        out.append(lat.get_populations())
        assert lat.sync()[1] == 0
        lat.close()
    assert torch.equal(out[0], out[1])
