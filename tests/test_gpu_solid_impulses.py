"""A channel only as high as the stencil is wide cannot hold a moving particle
inside the band the stencil needs, so part of its impulse falls on the solid planes.  It
belongs to the call that spread it: after the step it is gone, as the
impulses of fluid nodes are."""
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [11, 12, 256])
@pytest.mark.parametrize("dtype,equilibrium", [(L.LB_F32, 0), (L.LB_F16, 0), (L.LB_F32, 1)])
@pytest.mark.parametrize("kernel,overlap", [(2, False), (2, True), (3, True), (4, False), (4, True)])
@pytest.mark.parametrize("sums", [False, True])
def test_solid_planes_are_cleared(nx, dtype, equilibrium, kernel, overlap, sums):
    if equilibrium and sums:
        pytest.skip("the sums come from the quadratic update")
    shape, mid = (nx, 9, kernel + 1), 0.5 * kernel  # the band is the one plane z = mid
    lat = L.Lattice(shape, kT=0.0, walls=True, dtype=dtype, equilibrium=equilibrium)
    facc = torch.empty((3,) + shape[::-1], dtype=torch.float32, device="cuda")
    out = torch.empty(38, dtype=torch.float64, device="cuda")

    def couple(overlap):
        lat.init_equilibrium()
        # near the ends of a row and of a plane, so that stencils wrap
        pos = torch.tensor([[0.2, 0.3, mid], [nx - 0.4, 8.6, mid]], dtype=torch.float64).cuda()
        mom = torch.tensor([[0.05, -0.02, 0.04], [0.01, 0.03, -0.06]], dtype=torch.float32).cuda()
        parts = L.particles(2, pos, mom, gamma0=2.0)
        L.lb_couple_particles(lat.h, parts, L.couple_params(n_substeps=1, dt=0.1, kernel=kernel, overlap=overlap))

    couple(False)
    L.lb_get_particle_forces(lat.h, facc)
    first = facc.clone()
    assert first[:, [0, -1]].abs().max() > 0
    for _ in range(2):
        lat.step(1) if not sums else L.lb_step_sums(lat.h, 1, out)
        couple(overlap)
        lat.step(1) if not sums else L.lb_step_sums(lat.h, 1, out)
        couple(False)
        L.lb_get_particle_forces(lat.h, facc)
        assert torch.equal(facc, first)
    assert lat.sync()[1] == 0
    lat.close()
