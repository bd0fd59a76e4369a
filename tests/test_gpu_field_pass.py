"""The pass that forms initial populations and auxiliary fields (F, P, the
chemical potentials) from the densities."""
import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_lattice_of_more_tile_rows_than_a_grid_dimension():
    """65536 and more tiles along y (a grid's second dimension ends at 65535)."""
    from paper_1904_06881_gb300 import tlb

    nx, ny, nz = 3, 4 * 65536 + 5, 3
    lat = tlb.Lattice(W.D3Q27, nx, ny, nz, **W.base_params())
    rho = np.full((nz, ny, nx), W.RHO_L)
    rho[:, ny - 40:, :] = 1.01 * W.RHO_L       # the far end is formed too
    lat.init_fields(rho, np.zeros_like(rho))
    f = lat.fields()
    assert np.abs(f["rho"] - rho).max() <= 1e-6 * W.RHO_L
    lat.step(2)
    lat.sync()
    assert np.abs(lat.aux("Fy")[:, ny - 45:]).max() > 1e-3
    assert np.abs(lat.aux("Fy")[:, 50:ny - 100]).max() <= 1e-6
    lat.close()


@pytest.mark.parametrize("eos", [0, 1, 2])
@pytest.mark.parametrize("size", [(W.D2Q9, 70, 40, 1), (W.D3Q27, 36, 20, 18)])
def test_auxiliary_force_is_that_of_the_step(eos, size):
    """A fluid at rest near rho = 1, whose stored populations f - w are small: the momentum
    that one step gives a node is its force, to the rounding of those."""
    from paper_1904_06881_gb300 import tlb

    lattice, nx, ny, nz = size
    lat = tlb.Lattice(lattice, nx, ny, nz, **W.base_params(rho_g=W.RHO_L / 10.0, eos=eos))
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(np.float64)
    two_pi = 2 * np.pi
    wave = np.sin(two_pi * x / nx + 0.3) + np.cos(two_pi * y / ny + 0.7) + (np.sin(two_pi * z / nz) if nz > 1 else 0.0)
    c, w = tlb.tlb_lattice_directions(lattice)
    rho, phi = 1.0 + 1e-3 * wave, 0.3 * np.cos(two_pi * x / nx) * np.ones_like(wave)
    lat.set_populations(w[:, None] * rho.reshape(1, -1), w[:, None] * phi.reshape(1, -1))
    F = [lat.aux(k) for k in ("Fx", "Fy", "Fz")[:lat.D]]
    lat.step(1)
    f = lat.populations()[0]
    lat.sync()
    w32 = np.ones(lat.Q, np.float32)           # the weights as the library forms them
    for a in range(lat.D):
        w32 = w32 * np.where(c[:, a] == 0, np.float32(2) / np.float32(3), np.float32(1) / np.float32(6))
    stored = f - w32.astype(np.float64)[:, None]
    j = np.zeros((lat.D,) + lat.shape)
    for i in range(lat.Q):                     # back to the node that it was streamed from
        fi = np.roll(stored[i].reshape(lat.shape), [-c[i, 2], -c[i, 1], -c[i, 0]], (0, 1, 2))
        for a in range(lat.D):
            j[a] += c[i, a] * fi
    # half a unit in the last place of each moving population, and as much again twice
    # over for the sums that close the momentum balance
    tol = 3 * lat.Q * 2.0 ** -24 * np.abs(stored[1:]).max()
    for a in range(lat.D):
        assert np.abs(F[a]).max() > 1e3 * tol
        assert np.abs(j[a] - F[a]).max() <= tol, (a, np.abs(j[a] - F[a]).max(), tol)
    lat.close()
