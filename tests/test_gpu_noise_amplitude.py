"""The noise amplitude over the whole range of temperatures a box may have:
the standard deviation sqrt(mu rho) multiplies the unit Gaussians after their
radius is formed, so temperatures whose variance times -2 ln v would be
denormal in FP32 still give the oracle's noise."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(8, 6, 5), (7, 6, 5)])  # paired and single nodes
@pytest.mark.parametrize("kT", [1e-36, 1e-20, 1e-4])
def test_noise_amplitude(ora, shape, kT):
    from paper_0803_2826_gb300 import lbfluct as L
    lat = L.Lattice(shape, kT=kT, seed=11)
    lat.init_equilibrium()
    lat.step(1)
    cur, _ = L.lb_state_buffers(lat.h)
    buf = [b for b in lat._bufs if b.data_ptr() == cur][0]
    n = shape[0] * shape[1] * shape[2]
    dev = buf.view(torch.float32).view(19, -1)[:, :n].double().cpu().numpy()
    # from rest the step leaves the noise alone: sqrt(kT) times that of kT = 1
    p = ora.make_params(shape, kT=1e-4, seed=11)
    rest = ora.equilibrium(p, None, None)
    want = (ora.step(p, rest, None, 0) - rest).reshape(19, n) * np.sqrt(kT / 1e-4)
    # the Gaussians are good to the hardware log2 (1.7e-6 of a radius) and sine
    # (2^-21 of it), summed over 15 modes: below 5e-6 of the largest deviation
    assert np.abs(dev - want).max() <= 5e-6 * np.abs(want).max()
    lat.close()
