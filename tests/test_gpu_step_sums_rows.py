"""lb_step_sums on rows of odd length: pairs that straddle rows and planes, the
lone last node, channels whose first pair holds a solid node.  The sums are
those of lb_moments, the populations those of lb_step."""
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 3), (1, 1, 4), (3, 3, 3), (5, 7, 4), (1, 64, 9), (3, 200, 5), (65, 3, 4), (127, 2, 3), (257, 5, 3)])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("dtype", [L.LB_F32, L.LB_BF16])
def test_odd_rows(shape, walls, dtype):
    field = torch.as_tensor(inputs.gaussian_field(shape, 3, 1e-4, seed=3), dtype=torch.float32).cuda()
    lats = [L.Lattice(shape, kT=1e-4, seed=5, walls=walls, dtype=dtype, force=field) for _ in range(2)]
    u = torch.as_tensor(inputs.gaussian_field(shape, 3, 1e-2, seed=4)).cuda()
    got, want = (torch.empty(38, dtype=torch.float64, device="cuda") for _ in range(2))
    for lat in lats:
        lat.init_equilibrium(None, u)
        lat.step(1)
    for _ in range(2):
        L.lb_moments(lats[1].h, None, None, None, want)
        L.lb_step_sums(lats[0].h, 1, got)
        lats[1].step(1)
        assert torch.equal(lats[0].get_populations(), lats[1].get_populations())
        n = shape[0] * shape[1] * (shape[2] - 2 * walls)
        # a block adds 256 nodes in FP32: at most 256 roundings of sum |x| <= sqrt(N sum x^2); blocks compensated
        tol = torch.cat([(n * want[19:]).sqrt(), want[19:]]) * 2.0 ** -16
        assert ((got - want).abs() <= tol).all(), (got - want).abs() / tol
    for lat in lats:
        assert lat.sync()[1] == 0
        lat.close()
