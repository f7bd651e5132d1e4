"""Several lanes a particle in the overlapped order: the stencil records they
leave reach every node they spread to (the step's populations are those of the
serial order), on both sides of the counts and box sizes where the form
changes, with masses and frictions of each particle and three-point noise."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu
KT = 1e-4


def _positions(n, shape, seed):
    per = [int(s / 1.3) for s in shape]
    k = np.arange(n)
    grid = np.stack([k % per[0], k // per[0] % per[1], k // (per[0] * per[1])], 1)
    assert grid[:, 2].max() < per[2]
    return (grid + 0.5) * 1.3 + np.random.default_rng(seed).uniform(-0.1, 0.1, (n, 3))


def _run(shape, n, kernel, overlap, dtype, per_particle, noise_kind, steps=2):
    lat = L.Lattice(shape, kT=KT, seed=3, dtype=dtype)
    lat.init_equilibrium()
    pos = torch.as_tensor(_positions(n, shape, 4)).cuda()
    mom = torch.as_tensor(inputs.maxwell_momenta(n, 1.0, KT, seed=5), dtype=torch.float32).cuda()
    rng = np.random.default_rng(6)
    kw = {}
    if per_particle:
        kw = {k: torch.as_tensor(rng.uniform(lo, 2.0 * lo, n), dtype=torch.float32).cuda() for k, lo in (("mass", 1.0), ("gamma", 1.5))}
    parts = L.particles(n, pos, mom, gamma0=2.0, **kw)
    out = []
    for t in range(steps):
        cp = L.couple_params(n_substeps=6, dt=0.1, seed=5, md_step0=6 * t, use_wca=True, eps=0.01, kernel=kernel,
                             overlap=overlap, noise_kind=noise_kind, fext=(1e-2, 0, -1e-2))
        L.lb_couple_particles(lat.h, parts, cp)
        lat.step(1)  # (no query in between: it would join the overlap)
        out.append((lat.get_populations(), pos.clone(), mom.clone()))
    assert lat.sync()[1] == 0
    lat.close()
    return out


# 1216 / 1217: a warp, eight lanes; 7296 / 7297: three blocks of 16 particles on 152 SMs and one more;
# 2432 / 2433 in boxes of more than 2^22 nodes: eight lanes, with phi_4 one thread
@pytest.mark.parametrize("kernel", [3, 4])
@pytest.mark.parametrize("shape,n,dtype,per_particle,noise_kind",
                         [((48, 46, 50), 1216, L.LB_F32, True, 1), ((48, 46, 50), 1217, L.LB_F32, True, 0),
                          ((48, 46, 50), 7296, L.LB_F32, False, 0), ((48, 46, 50), 7297, L.LB_F32, True, 1),
                          ((48, 46, 50), 2500, L.LB_F16, False, 1), ((47, 46, 50), 2500, L.LB_BF16, True, 0),
                          ((168, 160, 160), 2432, L.LB_F32, False, 0), ((168, 160, 160), 2433, L.LB_F32, False, 0)])
def test_against_serial(shape, n, dtype, per_particle, noise_kind, kernel):
    got = _run(shape, n, kernel, True, dtype, per_particle, noise_kind)
    want = _run(shape, n, kernel, False, dtype, per_particle, noise_kind)
    # the first call starts from equal states and every form moves a particle alike, bit for bit
    assert torch.equal(got[0][1], want[0][1]) and torch.equal(got[0][2], want[0][2])
    # deviations are thermal, below 2^-4 (six times 1e-2).  FP32: the correction of the stored result and the
    # order of the impulse atomics, eight units in the last place of 2^-5; 16 bits: a unit of the stored
    # value (below 64), 2^5 2^-10 or 2^5 2^-7 over the scale 2^10; twice that a step, for what it moves in the next
    unit = {L.LB_F32: 2.0 ** -25, L.LB_F16: 2.0 ** -15, L.LB_BF16: 2.0 ** -12}[dtype]
    for t, (x, y) in enumerate(zip(got, want)):
        assert (x[0] - y[0]).abs().max().item() <= 2 * (t + 1) * unit
