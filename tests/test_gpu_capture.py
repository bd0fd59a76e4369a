"""tlb_step on a stream that is recorded into a CUDA graph: the replayed steps
take the solid mask that is set when they run, not the one of the recording,
and a recording that has been invalidated refuses steps, which then do not
count.  tlb_step_noalloc is recorded with its geometry's flags in place only."""
import ctypes

import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _wl(lattice, mask_kind):
    nx, ny, nz = (96, 40, 1) if lattice == W.D2Q9 else (32, 16, 12)
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(np.float64)
    d2 = (x - 0.45 * nx) ** 2 + (y - 0.5 * ny) ** 2 + (0.0 if nz == 1 else (z - 0.5 * nz) ** 2)
    C2 = 0.5 * (1.0 - np.tanh((np.sqrt(d2) - 5.0) / 2.0))
    rho, phi = W.phase_fields(C2, np.zeros_like(C2))
    mask = np.zeros((nz, ny, nx), np.uint8)
    if mask_kind == "block":
        mask[: min(nz, 5), 3:9, nx - 9:nx - 4] = 1
    return dict(name="capture", lattice=lattice, nx=nx, ny=ny, nz=nz, mask=mask, rho=rho, phi=phi,
                params=W.base_params(wetting=W.WET_FORCE, kw_rho=0.05))


class _Driver:
    """The driver's stream capture, for a stream given as an integer handle."""

    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")

    def begin(self, stream):
        assert self.cu.cuStreamBeginCapture_v2(ctypes.c_void_p(stream), 1) == 0        # this thread's calls only

    def end(self, stream):
        graph = ctypes.c_void_p()
        return self.cu.cuStreamEndCapture(ctypes.c_void_p(stream), ctypes.byref(graph)), graph

    def instantiate(self, graph):
        ex = ctypes.c_void_p()
        assert self.cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)) == 0
        return ex

    def launch(self, ex, stream):
        assert self.cu.cuGraphLaunch(ex, ctypes.c_void_p(stream)) == 0

    def destroy(self, graph, ex):
        self.cu.cuGraphExecDestroy(ex)
        self.cu.cuGraphDestroy(graph)


@pytest.mark.parametrize("lattice", [W.D2Q9, W.D3Q27])
def test_recorded_steps_follow_a_new_mask(lattice):
    import torch

    from paper_1904_06881_gb300 import tlb

    drv = _Driver()
    open_, block = _wl(lattice, "none"), _wl(lattice, "block")
    s = torch.cuda.Stream()
    lat = tlb.lattice_from_workload(open_)
    lat.step(2)
    lat.sync()
    tlb.tlb_set_stream(lat.h, s.cuda_stream)
    drv.begin(s.cuda_stream)
    tlb.tlb_step(lat.h, 4)                     # an even number: the buffers' roles return
    rc, graph = drv.end(s.cuda_stream)
    assert rc == 0
    ex = drv.instantiate(graph)
    for wl in (block, open_, block):
        lat.set_solid(wl["mask"])
        lat.init_fields(wl["rho"], wl["phi"])
        drv.launch(ex, s.cuda_stream)
        torch.cuda.synchronize()
        ref = tlb.lattice_from_workload(wl)
        ref.step(4)
        fl = wl["mask"].reshape(-1) == 0
        for a, b in zip(lat.populations(), ref.populations()):
            assert np.array_equal(a[:, fl], b[:, fl])
        ref.close()
    drv.destroy(graph, ex)
    lat.close()


@pytest.mark.parametrize("lattice", [W.D2Q9, W.D3Q27])
@pytest.mark.parametrize("phases", [False, True])
def test_steps_that_cannot_be_launched_do_not_count(lattice, phases):
    import torch

    from paper_1904_06881_gb300 import tlb

    drv, wl, s = _Driver(), _wl(lattice, "block"), torch.cuda.Stream()
    lat, ref = tlb.lattice_from_workload(wl), tlb.lattice_from_workload(wl)
    for l in (lat, ref):
        l.step(3)
        l.sync()
    tlb.tlb_set_stream(lat.h, s.cuda_stream)
    drv.begin(s.cuda_stream)
    assert tlb.lib().tlb_sync(lat.h) == -3     # a synchronisation, which ends the recording
    for _ in range(3):                         # an odd number of steps refused
        rc = tlb.lib().tlb_step_phase(lat.h, 2) if phases else tlb.lib().tlb_step(lat.h, 1)
        assert rc == -3
    assert drv.end(s.cuda_stream)[0] != 0
    assert lat.steps_done == 3
    for l in (lat, ref):
        l.step(4)
        l.sync()
    assert lat.steps_done == 7
    fl = wl["mask"].reshape(-1) == 0
    for a, b in zip(lat.populations(), ref.populations()):
        assert np.array_equal(a[:, fl], b[:, fl])
    lat.close()
    ref.close()


@pytest.mark.parametrize("lattice", [W.D2Q9, W.D3Q27])
def test_recorded_allocation_free_steps(lattice):
    import torch

    from paper_1904_06881_gb300 import tlb

    drv, wl, s = _Driver(), _wl(lattice, "block"), torch.cuda.Stream()
    ref = tlb.lattice_from_workload(wl)
    c, _ = tlb.tlb_lattice_directions(lattice)
    w = np.ones(len(c), np.float32)            # the weights as the library forms them
    for a in range(2 if lattice == W.D2Q9 else 3):
        w = w * np.where(c[:, a] == 0, np.float32(2) / np.float32(3), np.float32(1) / np.float32(6))
    w = w.astype(np.float64)[:, None]
    f0, g0 = ref.populations()
    f, g = (torch.tensor(v.astype(np.float32), device="cuda") for v in (f0 - w, g0))
    f_tmp, g_tmp = torch.empty_like(f), torch.empty_like(g)
    torch.cuda.synchronize()
    p = tlb.make_params(lattice, wl["nx"], wl["ny"], wl["nz"], **wl["params"])

    def call(nsteps):
        tlb.tlb_step_noalloc(p, wl["mask"], f.data_ptr(), f_tmp.data_ptr(), g.data_ptr(), g_tmp.data_ptr(), nsteps,
                             s.cuda_stream)

    drv.begin(s.cuda_stream)
    with pytest.raises(tlb.TlbError) as e:
        call(3)
    assert e.value.code == -4
    rc, graph = drv.end(s.cuda_stream)         # the recording itself stays valid
    assert rc == 0
    drv.cu.cuGraphDestroy(graph)
    call(0)
    drv.begin(s.cuda_stream)
    call(3)
    rc, graph = drv.end(s.cuda_stream)
    assert rc == 0
    ex = drv.instantiate(graph)
    fl = wl["mask"].reshape(-1) == 0
    for _ in range(2):
        drv.launch(ex, s.cuda_stream)
        torch.cuda.synchronize()
        ref.step(3)
        fr, gr = ref.populations()
        assert np.array_equal((f.double().cpu().numpy() + w)[:, fl], fr[:, fl])
        assert np.array_equal(g.double().cpu().numpy()[:, fl], gr[:, fl])
    drv.destroy(graph, ex)
    ref.close()
