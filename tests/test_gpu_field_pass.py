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
