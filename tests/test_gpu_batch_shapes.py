"""Launch shapes of the batched kernel: which block sizes run, and that the
result does not depend on them."""
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu
ODD, EVEN = [(7, 5, 9), (8, 6, 5), (33, 4, 3)], [(8, 6, 5), (64, 3, 2), (34, 4, 3)]


def _run(shapes, threads, dtype, kT, records, steps=3):
    stream = torch.cuda.Stream()
    B = L.Batch(shapes, seeds=[21 + k for k in range(len(shapes))], dtype=dtype, stream=stream, kT=kT)
    rec = torch.empty((len(shapes), steps, 12), dtype=torch.float64, device="cuda")
    try:
        with torch.cuda.stream(stream):
            if records:
                L.lb_batch_record_modes(B.b, rec, steps)
            L.lb_batch_set_config(B.b, threads, 64, 1)
            for k, s in enumerate(shapes):
                L.lb_batch_init_equilibrium(B.b, k, None, torch.as_tensor(inputs.gaussian_field(s, 3, 1e-2, seed=30 + k)).cuda())
            L.lb_batch_step(B.b, steps, False)
        L.lb_batch_sync(B.b)
        return [B.get_populations(k) for k in range(len(shapes))], rec
    finally:
        B.close()


@pytest.mark.parametrize("dtype", [L.LB_F32, L.LB_F16, L.LB_BF16])
@pytest.mark.parametrize("kT", [0.0, 1e-4])
@pytest.mark.parametrize("records", [False, True])
def test_shapes_that_run(dtype, kT, records):
    cases = [(ODD, t) for t in (512, 544, 640, 896, 1024)] + [(EVEN, 512)]
    want = {id(s): _run(s, 64, dtype, kT, records) for s in (ODD, EVEN)}
    for shapes, threads in cases:
        pops, rec = _run(shapes, threads, dtype, kT, records)
        w = want[id(shapes)]
        assert all(torch.equal(x, y) for x, y in zip(pops, w[0])), (shapes, threads)
        if records:
            # FP32 sums of at most 384 velocities of order 1e-2, grouped by warps and added in any order
            assert (rec - w[1]).abs().max().item() < 384 * 1e-2 * 2.0 ** -22


def test_shapes_that_are_refused():
    for shapes, threads, status in ((EVEN, 1024, L.LB_EUNSUPPORTED), (EVEN, 640, L.LB_EUNSUPPORTED), (ODD, 1056, L.LB_EINVAL),
                                    (ODD, 48, L.LB_EINVAL), (ODD, 0, L.LB_EINVAL)):
        with pytest.raises(L.LBError) as e:
            _run(shapes, threads, L.LB_F32, 1e-4, False)
        assert e.value.status == status
