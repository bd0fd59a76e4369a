"""Densities that an equation of state does not admit are reported: van der
Waals and Peng-Robinson end at rho = 1/b, where their pressure has its pole
and their free energy the logarithm's, so a state beyond it has diverged."""
import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _uniform(lat, rho):
    """Populations at rest of the density field rho (per node), phi = 0."""
    from paper_1904_06881_gb300 import tlb

    _, w = tlb.tlb_lattice_directions(lat.lattice)
    lat.set_populations(w[:, None] * rho.reshape(1, -1), np.zeros((lat.Q, lat.N)))


@pytest.mark.parametrize("eos", [1, 2])
@pytest.mark.parametrize("size", [(W.D2Q9, 40, 20, 1), (W.D3Q27, 20, 9, 8)])
@pytest.mark.parametrize("walls", [0, 1])
def test_density_beyond_the_pole_is_reported(eos, size, walls):
    from paper_1904_06881_gb300 import tlb

    lat = tlb.Lattice(*size, **W.base_params(rho_g=W.RHO_L / 10.0, eos=eos))
    if walls:
        mask = np.zeros(lat.shape, np.uint8)
        mask[:, 0] = 1
        lat.set_solid(mask)
    limit = 1.0 / lat.derived["b"]
    _uniform(lat, np.full(lat.N, 0.9 * limit))
    lat.step(1)
    lat.sync()                                 # admitted: nothing to report
    beyond = np.full(lat.N, 1.2 * limit)
    one = np.full(lat.N, 0.9 * limit)
    one[lat.N // 2 + 3] = 1.2 * limit          # its neighbours feel its pressure
    for rho in (beyond, one):
        _uniform(lat, rho)
        lat.step(1)
        with pytest.raises(tlb.TlbError) as e:
            lat.sync()
        assert e.value.code == -6
        lat.init_fields(np.full(lat.shape, W.RHO_L), np.zeros(lat.shape))      # takes the error back
    lat.close()
