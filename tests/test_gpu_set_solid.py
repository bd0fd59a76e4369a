"""tlb_set_solid that fails leaves the context as it was."""
import ctypes

import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(W.D2Q9, 96, 40, 1), (W.D3Q27, 32, 16, 12)])
def test_failed_allocation_keeps_the_former_mask(size):
    from paper_1904_06881_gb300 import tlb

    lattice, nx, ny, nz = size
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(np.float64)
    C2 = 0.5 * (1.0 - np.tanh((np.hypot(x - 0.4 * nx, y - 0.5 * ny) - 6.0) / 2.0))
    rho, phi = W.phase_fields(C2, np.zeros_like(C2))
    wall = np.zeros((nz, ny, nx), np.uint8)
    wall[:, 0] = 1
    more = wall.copy()
    more[:, ny - 1] = 1                        # a longer ghost list: a new block for it
    more[:, 8:14, nx - 12:nx - 5] = 1
    wl = dict(name="mask", lattice=lattice, nx=nx, ny=ny, nz=nz, mask=wall, rho=rho, phi=phi,
              params=W.base_params(wetting=W.WET_GEOM_EXTRAP, theta_deg=(70.0, 70.0, 90.0)))
    lat, ref = tlb.lattice_from_workload(wl), tlb.lattice_from_workload(wl)
    lat.step(4)
    ref.step(4)
    ALLOC = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
    FREE = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)
    a, f = ALLOC(lambda nbytes, user: None), FREE(lambda ptr, user: None)
    assert tlb.lib().tlb_set_allocator(ctypes.cast(a, ctypes.c_void_p), ctypes.cast(f, ctypes.c_void_p), None) == 0
    try:
        with pytest.raises(tlb.TlbError) as e:
            lat.set_solid(more)
    finally:
        tlb.default_allocator()
    assert e.value.code == -2
    for again in (False, True):                # the steps go on, and new fields take the former mask too
        if again:
            lat.init_fields(rho, phi)
            ref.init_fields(rho, phi)
        lat.step(5)
        ref.step(5)
        fl = wall.reshape(-1) == 0
        for p, q in zip(lat.populations(), ref.populations()):
            assert np.array_equal(p[:, fl], q[:, fl])
        assert np.array_equal(lat.aux("rho_ghost"), ref.aux("rho_ghost"))
        assert np.array_equal(lat.fields()["rho"], ref.fields()["rho"])
    lat.close()
    ref.close()
