"""The ways by which a D3Q27 tile's populations reach shared memory (tensor copies,
words, pairs of halves, single halves), at row lengths on either side of each
rule, against the FP64 oracle and, in FP32, against tlb_step_noalloc, which has
no tensor copies; walls at every distance from a tile's edge along y and z; and
node offsets beyond 32 bits."""
import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

from helpers import gpu_from_workload, normwise, oracle_from_workload
from test_gpu_parity import _perturbed_oracle_spread

pytestmark = pytest.mark.gpu

STEPS = 5
# Five steps in FP32: a density is a sum of up to 27 populations that four
# operations a step round by 6e-8 of themselves, 1.5e-6 of rho_l = 6.1 or 2.6e-7
# of rho_l - rho_g a step at worst; the force feeds a few times that back.
TOL = 1e-5
# FP16 moving populations of g: the parity tests' bound (200 steps)
TOL_FP16 = 2e-5


def _mask(nx, ny, nz, kind):
    m = np.zeros((nz, ny, nx), np.uint8)
    if kind == "plane":
        m[0] = 1
    elif kind == "blocks":                      # two blocks, one across the periodic edges
        m[1:4, 1:3, 2:4] = 1
        m[np.ix_([nz - 1, 0], [ny - 1, 0], [nx - 1, 0])] = 1
    elif kind[0] in "yz":                       # a block whose near face lies `d` nodes behind y = 4 or z = 4
        o = 4 + int(kind[1:])
        m[(slice(o, o + 2), slice(2, 5)) if kind[0] == "z" else (slice(2, 5), slice(o, o + 2))] = 1
        m[:, :, nx // 2:] = 0                   # ... half as long as the lattice
    return m


def _wl(nx, ny, nz, kind, wetting=W.WET_FORCE, **params):
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(np.float64)
    R = 0.3 * min(nx, ny, nz)
    d = np.sqrt((x - 0.43 * nx - 0.3) ** 2 + (y - 0.52 * ny - 0.2) ** 2 + (z - 0.47 * nz - 0.1) ** 2)
    C2 = 0.5 * (1.0 - np.tanh((d - R) / 2.0))
    rho, phi = W.phase_fields(C2, np.random.default_rng(nx).uniform(-1e-3, 1e-3, C2.shape))
    p = W.base_params(wetting=wetting, **params)
    p.update(dict(kw_rho=0.05) if wetting == W.WET_FORCE else dict(theta_deg=(70.0, 70.0, 90.0)))
    return dict(name="staging", lattice=W.D3Q27, nx=nx, ny=ny, nz=nz, mask=_mask(nx, ny, nz, kind), rho=rho, phi=phi, params=p)


def _against_oracle(wl, tol, fp16=0):
    g, o = gpu_from_workload(wl, g_fp16=fp16), oracle_from_workload(wl)      # the oracle keeps g in FP64
    g.step(STEPS)
    o.step(STEPS)
    e = normwise(g.fields(), o.fields(), o.derived, mask=wl["mask"])
    g.close()
    for k in ("rho", "phi", "C"):
        assert e[k] <= (tol[k] if isinstance(tol, dict) else tol), (e, tol)


ROWS = [16, 17, 18, 19, 20, 24, 33, 34, 36, 40, 47]


@pytest.mark.parametrize("fp16", [0, 1])
@pytest.mark.parametrize("kind", ["none", "plane", "blocks"])
@pytest.mark.parametrize("nx", ROWS)
def test_rows_against_the_oracle(nx, kind, fp16):
    _against_oracle(_wl(nx, 9, 10, kind), TOL_FP16 if fp16 else TOL, fp16)


@pytest.mark.parametrize("kind", ["none", "blocks"])
@pytest.mark.parametrize("nx", ROWS)
def test_rows_with_and_without_tensor_copies(nx, kind):
    import torch

    from paper_1904_06881_gb300 import tlb

    wl = _wl(nx, 9, 10, kind)
    lat = gpu_from_workload(wl)
    c, _ = tlb.tlb_lattice_directions(wl["lattice"])
    w = np.ones(len(c), np.float32)             # the weights as the library forms them
    for a in range(3):
        w = w * np.where(c[:, a] == 0, np.float32(2) / np.float32(3), np.float32(1) / np.float32(6))
    w = w.astype(np.float64)[:, None]
    f0, g0 = lat.populations()
    f, g = (torch.tensor(v.astype(np.float32), device="cuda") for v in (f0 - w, g0))
    f_tmp, g_tmp = torch.empty_like(f), torch.empty_like(g)
    tlb.tlb_step_noalloc(tlb.make_params(wl["lattice"], nx, 9, 10, **wl["params"]), wl["mask"], f.data_ptr(),
                         f_tmp.data_ptr(), g.data_ptr(), g_tmp.data_ptr(), STEPS, torch.cuda.current_stream().cuda_stream)
    lat.step(STEPS)
    torch.cuda.synchronize()
    fl = wl["mask"].reshape(-1) == 0
    fr, gr = lat.populations()
    assert np.array_equal((f.double().cpu().numpy() + w)[:, fl], fr[:, fl])
    assert np.array_equal(g.double().cpu().numpy()[:, fl], gr[:, fl])
    lat.close()


@pytest.mark.parametrize("fp16", [0, 1])
@pytest.mark.parametrize("axis", ["y", "z"])
@pytest.mark.parametrize("d", [0, 1, 2, 3])
def test_blocks_along_y_and_z(axis, d, fp16):
    _against_oracle(_wl(24, 13, 14, "%s%d" % (axis, d), W.WET_GEOM_EXTRAP), TOL_FP16 if fp16 else TOL, fp16)


@pytest.mark.parametrize("kind", ["plane", "blocks", "y1", "z2"])
def test_interpolation_in_three_dimensions(kind):
    """The sample cell changes where a gradient's sign does: held to what the oracle
    itself reproduces under perturbations of its populations, as in the parity tests."""
    wl = _wl(24, 13, 14, kind, W.WET_GEOM_INTERP)
    _, spread = _perturbed_oracle_spread(wl, STEPS)
    _against_oracle(wl, {k: max(TOL, 3 * spread[k]) for k in ("rho", "phi", "C")})


def test_node_offsets_beyond_32_bits():
    """2^30 nodes and more: the same lattice over and over gives the bits of one of it."""
    import torch

    from paper_1904_06881_gb300 import tlb

    if torch.cuda.mem_get_info()[0] < 230 << 30:
        pytest.skip("needs 190 GB of device memory")
    bx, by, kx, ky = 256, 4097, 128, 8          # 32768 x 32776 nodes
    assert bx * by * kx * ky >= 1 << 30
    y, x = torch.meshgrid(torch.arange(by, dtype=torch.float64), torch.arange(bx, dtype=torch.float64), indexing="ij")
    C2 = 0.5 * (1.0 - torch.tanh((torch.hypot(x - 100.3, (y % 241) - 40.2) - 30.0) / 2.0))
    rho = (W.RHO_L * C2 + W.RHO_G * (1.0 - C2)).float()
    phi = (5.0 * C2).float()
    mask = np.zeros((by, bx), np.uint8)
    mask[0] = 1
    mask[2000:2003, 77:140] = 1
    fluid = torch.from_numpy(1 - mask)
    rho, phi = (rho * fluid).cuda(), (phi * fluid).cuda()
    small = tlb.Lattice(W.D2Q9, bx, by, 1, **W.base_params(wetting=W.WET_FORCE, kw_rho=0.05))
    small.set_solid(mask)
    tlb.tlb_init_fields_device(small.h, rho.data_ptr(), phi.data_ptr())
    small.step(4)
    out = [torch.empty_like(rho) for _ in range(2)]
    tlb.tlb_get_fields_device(small.h, *(t.data_ptr() for t in out))
    small.sync()
    big = tlb.Lattice(W.D2Q9, bx * kx, by * ky, 1, **W.base_params(wetting=W.WET_FORCE, kw_rho=0.05))
    big.set_solid(np.tile(mask, (ky, kx)))
    many = [t.repeat(ky, kx) for t in (rho, phi)]
    tlb.tlb_init_fields_device(big.h, many[0].data_ptr(), many[1].data_ptr())
    big.step(4)
    tlb.tlb_get_fields_device(big.h, many[0].data_ptr(), many[1].data_ptr())
    big.sync()
    for t, o in zip(many, out):
        for k in range(ky):
            rows = t[k * by:(k + 1) * by].view(by, kx, bx)
            assert all(torch.equal(rows[:, j], o) for j in range(kx))
    big.close()
    small.close()
