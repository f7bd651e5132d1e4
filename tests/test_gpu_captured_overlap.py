"""Overlapped coupled steps recorded in a CUDA graph: the re-update of impulse
nodes is launched as a chain behind an event of the coupling's stream."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_0803_2826_gb300 import inputs  # noqa: E402
from paper_0803_2826_gb300 import lbfluct as L  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [L.LB_F32, L.LB_F16])
@pytest.mark.parametrize("kernel", [2, 3, 4])
def test_captured(dtype, kernel):
    shape, n = (24, 22, 20), 48

    def go(graph):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            lat = L.Lattice(shape, kT=1e-4, seed=3, dtype=dtype, stream=stream)
            lat.init_equilibrium()
            pos = torch.as_tensor(inputs.random_walk_chains(2, n // 2, shape, seed=1)).cuda()
            mom = torch.as_tensor(inputs.maxwell_momenta(n, 1.0, 1e-4, seed=2), dtype=torch.float32).cuda()
            parts = L.particles(n, pos, mom, gamma0=2.0)

            def steps(t0, t1):
                for t in range(t0, t1):
                    cp = L.couple_params(n_substeps=4, dt=0.1, seed=5, md_step0=4 * t, chain_len=n // 2, use_wca=True,
                                         eps=0.01, k_fene=0.3, r0=1.5, kernel=kernel, overlap=True)
                    L.lb_couple_particles(lat.h, parts, cp)
                    lat.step(1)

            steps(0, 2)  # allocates, and builds the list once
            torch.cuda.synchronize()
            if graph:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=stream):
                    steps(2, 5)
                g.replay()
            else:
                steps(2, 5)
            torch.cuda.synchronize()
            out = lat.get_populations().cpu().numpy(), pos.cpu().numpy(), mom.cpu().numpy()
        assert lat.sync()[1] == 0
        lat.close()
        return out

    for k, (x, y) in enumerate(zip(go(True), go(False))):
        # the impulse atomics add in any order: FP32 rounding grown over five steps, and in FP16 a stored unit of
        # deviations below 2^-4 (2^-15) a step
        tol = 2e-5 * np.abs(y).max() if k or dtype == L.LB_F32 else 5 * 2.0 ** -15
        assert np.abs(x - y).max() < tol
