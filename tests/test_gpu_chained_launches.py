"""Kernels of a stream launched as a chain may start before their predecessor
ends; what they compute must not depend on it.  Steps issued back to back,
with other work of the stream in between, against the same steps with the
device waited for after every call, and inside a captured graph."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu


def _run(shape, wait, steps=40, **kw):
    field = torch.zeros(3, *shape[::-1], device="cuda")
    lat = L.Lattice(shape, force=field, seed=3, **kw)
    lat.init_equilibrium(None, torch.as_tensor(inputs.shear_wave(shape, 0.02)).cuda())
    for t in range(steps):
        field.fill_(1e-5 * (t % 3))  # the stream's own work between the steps
        lat.step(1 + t % 2)
        if wait:
            torch.cuda.synchronize()
    n = lat.get_populations()
    lat.sync()
    lat.close()
    return n


@pytest.mark.parametrize("shape,kw", [((16, 16, 16), {"kT": 1e-4}), ((64, 64, 64), {"kT": 1e-4}), ((33, 20, 17), {"kT": 1e-4}),
                                      ((61, 47, 31), {"kT": 0.0, "walls": True}), ((256, 64, 40), {"kT": 1e-4}),
                                      ((40, 30, 20), {"kT": 1e-4, "dtype": L.LB_F16}),
                                      ((40, 30, 20), {"kT": 1e-4, "equilibrium": 1})])
def test_back_to_back(shape, kw):
    assert torch.equal(_run(shape, False, **kw), _run(shape, True, **kw))


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("kernel", [2, 4])
def test_coupled_back_to_back(overlap, kernel):
    shape, n = (24, 22, 20), 48

    def go(wait):
        lat = L.Lattice(shape, kT=1e-4, seed=3)
        lat.init_equilibrium()
        pos = torch.as_tensor(inputs.random_walk_chains(2, n // 2, shape, seed=1)).cuda()
        mom = torch.as_tensor(inputs.maxwell_momenta(n, 1.0, 1e-4, seed=2), dtype=torch.float32).cuda()
        parts = L.particles(n, pos, mom, gamma0=2.0)
        for t in range(20):
            cp = L.couple_params(n_substeps=4, dt=0.1, seed=5, md_step0=4 * t, chain_len=n // 2, use_wca=True, eps=0.01,
                                 k_fene=0.3, r0=1.5, kernel=kernel, overlap=overlap)
            L.lb_couple_particles(lat.h, parts, cp)
            lat.step(1)
            if wait:
                torch.cuda.synchronize()
        pops = lat.get_populations()
        assert lat.sync()[1] == 0
        lat.close()
        return pops.cpu().numpy(), pos.cpu().numpy(), mom.cpu().numpy()

    for x, y in zip(go(False), go(True)):
        # the impulse atomics add in any order: FP32 rounding, grown over 20 steps
        assert np.abs(x - y).max() < 2e-5 * np.abs(y).max()


def test_spheres_back_to_back():
    shape = (32, 30, 28)

    def go(wait):
        lat = L.Lattice(shape, kT=1e-4, seed=3)
        lat.init_equilibrium()
        pos = torch.tensor([[8.0, 8.3, 7.9], [20.2, 19.0, 18.6]], dtype=torch.float64).cuda()
        vel = torch.tensor([[0.02, -0.01, 0.03], [-0.02, 0.03, 0.01]], dtype=torch.float64).cuda()
        sph = L.spheres(2, pos, vel, 3.0, mass0=100.0)
        L.lb_spheres_place(lat.h, sph)
        for _ in range(20):
            L.lb_step_spheres(lat.h, sph)
            if wait:
                torch.cuda.synchronize()
        assert lat.sync()[1] == 0
        own = torch.empty(shape[::-1], dtype=torch.int32, device="cuda")
        L.lb_get_solid_map(lat.h, own)
        pops = lat.get_populations() * (own < 0)
        lat.close()
        return pops.cpu().numpy(), pos.cpu().numpy(), vel.cpu().numpy()

    for x, y in zip(go(False), go(True)):
        assert np.abs(x - y).max() < 2e-5 * np.abs(y).max()


@pytest.mark.parametrize("shape,kw", [((32, 32, 32), {}), ((31, 9, 8), {"walls": True}), ((32, 32, 32), {"equilibrium": 1})])
def test_captured(shape, kw):
    """Steps recorded in a CUDA graph and replayed once are the steps issued directly."""
    stream = torch.cuda.Stream()
    want = L.Lattice(shape, kT=1e-4, seed=7, **kw)
    want.init_equilibrium()
    want.step(5)
    with torch.cuda.stream(stream):
        lat = L.Lattice(shape, kT=1e-4, seed=7, stream=stream, **kw)
        lat.init_equilibrium()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        lat.step(5)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(lat.get_populations(), want.get_populations())
    lat.close()
    want.close()
