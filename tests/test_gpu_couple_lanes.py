"""The persistent couplings (a warp, eight lanes or one thread a particle, by
count and stencil) against one launch per sub-step, at the counts where the
form changes, with lists rebuilt inside the call, over calls that clear the
impulses of the one before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu
KT = 1e-4


def _run(shape, pos0, mom0, length, kernel, per_substep, walls, calls, overlap=False, wca=True):
    n = pos0.shape[0]
    lat = L.Lattice(shape, kT=KT, seed=3, walls=walls)
    u = inputs.shear_wave(shape, 0.02)
    lat.init_equilibrium(None, torch.as_tensor(u).cuda())
    pos = torch.as_tensor(pos0).cuda()
    mom = torch.as_tensor(mom0, dtype=torch.float32).cuda()
    parts = L.particles(n, pos, mom, gamma0=2.0)
    facc = torch.empty((3,) + shape[::-1], dtype=torch.float32, device="cuda")
    for t in range(calls):
        cp = L.couple_params(n_substeps=6, dt=0.1, seed=5, md_step0=6 * t, chain_len=length, use_wca=wca, eps=0.01,
                             k_fene=0.3, r0=1.5, kernel=kernel, per_substep=per_substep, overlap=overlap,
                             fext=(1e-4, 0, -1e-4))
        L.lb_couple_particles(lat.h, parts, cp)
        L.lb_get_particle_forces(lat.h, facc)
        if t + 1 < calls:
            lat.step(1)
    assert lat.sync()[1] == 0
    lat.close()
    return pos.cpu().numpy(), mom.cpu().numpy().astype(np.float64), facc.cpu().numpy().astype(np.float64)


# 16 x 76 = 1216 particles fill two blocks of warps per SM, 16 x 152 = 2432 one block of eights, 9728 the resident eights of the wide stencils
@pytest.mark.parametrize("kernel", [2, 3, 4])
@pytest.mark.parametrize("chains,length,edge,fast", [(1, 2, 12, 1.0), (5, 7, 24, 1.0), (5, 7, 24, 60.0), (76, 16, 40, 1.0), (77, 16, 40, 60.0),
                                                     (152, 16, 48, 1.0), (153, 16, 48, 60.0), (640, 16, 64, 1.0)])
def test_against_per_substep(chains, length, edge, fast, kernel):
    shape = (edge, edge - 2, edge + 1)
    n = chains * length
    pos = inputs.random_walk_chains(chains, length, shape, seed=4)
    mom = inputs.maxwell_momenta(n, 1.0, KT, seed=5)
    # fast: whole chains drift together, far enough to change cells and to ask for a new list inside the call
    mom = mom + np.repeat(inputs.maxwell_momenta(chains, 1.0, KT, seed=6) * (fast - 1.0) / 2, length, axis=0)
    calls = 2
    got = _run(shape, pos, mom, length, kernel, False, False, calls)
    want = _run(shape, pos, mom, length, kernel, True, False, calls)
    d = got[0] - want[0]
    d -= np.array(shape) * np.round(d / np.array(shape))
    # FP32 chain forces agree with the FP64 oracle to 1e-5 of the momenta a call; two forms, two calls
    assert np.abs(d).max() < 5e-6
    for x, y in zip(got[1:], want[1:]):
        assert np.linalg.norm(x - y) < 4e-5 * np.linalg.norm(y)
        assert np.abs(x - y).max() < 1e-4 * np.abs(y).max()


@pytest.mark.parametrize("kernel", [2, 3, 4])
def test_walls_and_overlap(kernel):
    shape, chains, length = (24, 22, 20), 6, 4
    # straight chains along x (no bond across the walls), some against the band the walls reflect into
    pos = np.zeros((chains, length, 3))
    pos[:, :, 0] = 2.3 + 0.97 * np.arange(length)
    pos[:, :, 1] = 1.7 + 3.1 * np.arange(chains)[:, None]
    pos[:, :, 2] = np.linspace(2.05, shape[2] - 3.05, chains)[:, None]
    pos = pos.reshape(-1, 3)
    mom = inputs.maxwell_momenta(chains * length, 1.0, KT, seed=5)
    want = _run(shape, pos, mom, length, kernel, True, True, 3)
    for overlap in (False, True):
        got = _run(shape, pos, mom, length, kernel, False, True, 3, overlap)
        for x, y in zip(got, want):
            assert np.abs(x - y).max() < 1e-4 * np.abs(y).max()
