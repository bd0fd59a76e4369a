"""Steps whose launches overlap (each kernel starts before its predecessor has
finished and waits inside) give the bits of steps with the GPU drained in
between: nothing is read before it is written."""
import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

from helpers import gpu_from_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp16", [0, 1])
@pytest.mark.parametrize("size", [(W.D2Q9, 65, 33, 1), (W.D2Q9, 1024, 600, 1), (W.D3Q27, 33, 21, 18), (W.D3Q27, 96, 64, 64),
                                  (W.D3Q27, 101, 60, 60)])
def test_overlapped_steps_equal_separate_ones(size, fp16):
    lattice, nx, ny, nz = size
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(np.float64)
    C2 = 0.5 * (1.0 - np.tanh((np.hypot(x - 0.4 * nx, y - 0.5 * ny) - 0.2 * ny) / 2.0))
    rho, phi = W.phase_fields(C2, np.zeros_like(C2))
    mask = np.zeros((nz, ny, nx), np.uint8)
    mask[:, 0] = 1
    wl = dict(name="order", lattice=lattice, nx=nx, ny=ny, nz=nz, mask=mask, rho=rho, phi=phi,
              params=dict(W.base_params(wetting=W.WET_GEOM_EXTRAP, theta_deg=(70.0, 70.0, 90.0)), g_fp16=fp16))
    a, b = gpu_from_workload(wl), gpu_from_workload(wl)
    a.step(30)
    for _ in range(30):
        b.step(1)
        b.sync()
    for p, q in zip(a.populations(), b.populations()):
        assert np.array_equal(p, q)
    a.close()
    b.close()
