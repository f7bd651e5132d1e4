"""lb_adjoint_forward advances the state as lb_step would: it ends in the
buffer that as many steps end in, so a captured call with an even number of
steps continues from its own result when it is replayed."""
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu
SHAPE = (12, 9, 8)


def _lattice(stream=None):
    lat = L.Lattice(SHAPE, kT=0.0, force=torch.zeros(3, *SHAPE[::-1], device="cuda"), **({"stream": stream} if stream else {}))
    lat.init_equilibrium(None, torch.as_tensor(inputs.gaussian_field(SHAPE, 3, 1e-2, seed=4)).cuda())
    return lat


@pytest.mark.parametrize("before", [0, 1])
@pytest.mark.parametrize("steps", [1, 2, 3, 4, 7, 8])
@pytest.mark.parametrize("every", [1, 2, 3, 8])
def test_ends_where_steps_end(before, steps, every):
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    a, b = _lattice(), _lattice()
    for lat in (a, b):
        lat.step(before)
    start = L.lb_state_buffers(a.h)
    b.step(steps)
    L.lb_adjoint_forward(a.h, steps, every, (0, 0, 0), SHAPE, loss)
    assert L.lb_state_buffers(a.h) == (start if steps % 2 == 0 else start[::-1])
    assert torch.equal(a.get_populations(), b.get_populations())
    grad = torch.empty(3, *SHAPE[::-1], device="cuda")
    L.lb_adjoint_backward(a.h, grad)
    assert torch.isfinite(grad).all() and a.sync()[1] == 0
    a.close()
    b.close()


@pytest.mark.parametrize("before", [0, 1])
def test_replayed(before):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        lat = _lattice(stream)
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        L.lb_adjoint_forward(lat.h, 4, 2, (0, 0, 0), SHAPE, loss)  # allocates
        lat.step(before)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        L.lb_adjoint_forward(lat.h, 4, 2, (0, 0, 0), SHAPE, loss)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    want = _lattice()
    want.step(4 + before + 12)
    assert torch.equal(lat.get_populations(), want.get_populations())
    lat.close()
    want.close()
