"""A caller's allocator whose blocks do not lie on the boundaries of the widest
loads: the steps are the same, and a batch, whose tables cannot be read there,
is refused."""
import ctypes

import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

from helpers import gpu_from_workload

pytestmark = pytest.mark.gpu


class _Allocator:
    """torch's blocks, those that `shifted` picks by their size 4 bytes further on."""

    def __init__(self, shifted):
        import torch

        from paper_1904_06881_gb300 import tlb

        self.base = {}

        def alloc(nbytes, user):
            p = torch.cuda.caching_allocator_alloc(int(nbytes) + 256, torch.cuda.current_device())
            q = p + (4 if shifted(nbytes) else 0)
            self.base[q] = p
            return q

        def free(ptr, user):
            torch.cuda.caching_allocator_delete(self.base.pop(ptr))

        self.a = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)(alloc)
        self.f = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)(free)
        self.tlb = tlb

    def __enter__(self):
        assert self.tlb.lib().tlb_set_allocator(ctypes.cast(self.a, ctypes.c_void_p), ctypes.cast(self.f, ctypes.c_void_p),
                                                None) == 0
        return self

    def __exit__(self, *exc):
        self.tlb.default_allocator()


def _wl(nx, ny, nz):
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(np.float64)
    C2 = 0.5 * (1.0 - np.tanh((np.sqrt((x - 0.45 * nx) ** 2 + (y - 0.5 * ny) ** 2 + (z - 0.5 * nz) ** 2) - 5.0) / 2.0))
    rho, phi = W.phase_fields(C2, np.zeros_like(C2))
    return dict(name="alignment", lattice=W.D3Q27, nx=nx, ny=ny, nz=nz, mask=np.zeros((nz, ny, nx), np.uint8), rho=rho,
                phi=phi, params=W.base_params())


@pytest.mark.parametrize("nx", [40, 38, 37])
def test_rho_and_phi_off_an_8_byte_boundary(nx):
    """Lattices with tiles away from every edge, whose region is loaded in pairs where it can be."""
    wl = _wl(nx, 16, 16)
    ref = gpu_from_workload(wl)
    with _Allocator(lambda nbytes: nbytes == 4 * nx * 16 * 16) as alloc:
        lat = gpu_from_workload(wl)
        assert sum(q % 8 == 4 for q in alloc.base) == 2            # rho and phi
        lat.step(6)
        ref.step(6)
        for p, q in zip(lat.populations(), ref.populations()):
            assert np.array_equal(p, q)
        lat.close()
    ref.close()


def test_batch_tables_off_their_boundary_are_refused():
    from paper_1904_06881_gb300 import tlb

    wl = _wl(24, 12, 12)
    lats = [gpu_from_workload(wl) for _ in range(2)]
    lats[0].step(3)
    with _Allocator(lambda nbytes: True):
        with pytest.raises(tlb.TlbError) as e:
            tlb.Batch(lats)
        assert e.value.code == -1
        with pytest.raises(tlb.TlbError) as e:
            tlb.tlb_step_batch([l.h for l in lats], 3)
        assert e.value.code == -1
    assert [l.steps_done for l in lats] == [3, 0]
    tlb.tlb_step_batch([l.h for l in lats], 3)
    for l in lats:
        l.close()
