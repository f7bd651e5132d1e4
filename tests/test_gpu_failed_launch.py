"""A launch the GPU cannot take (more than 65535 blocks along y) is reported by
the call that made it and by no other."""
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sums", [False, True])
def test_error_is_reported_once(sums):
    lat = L.Lattice((256, 65536, 1), kT=0.0, dtype=L.LB_F16)
    lat.init_equilibrium()
    out = torch.empty(38, dtype=torch.float64, device="cuda")
    with pytest.raises(L.LBError) as e:
        L.lb_step_sums(lat.h, 1, out) if sums else lat.step(1)
    assert e.value.status == L.LB_ECUDA
    L.lb_moments(lat.h, None, None, None, out)
    lat.init_equilibrium()
    assert lat.sync()[1] == 0 and L.lb_get_step(lat.h) == 0
    lat.close()
