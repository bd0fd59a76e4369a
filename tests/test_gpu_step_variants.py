"""The forms that a step takes, at the sizes where they change: tiles with and
without solid nodes in reach (2 nodes), their flags as launch parameters (up to
1024 tiles) and from memory, populations staged by tensor copies, in 16-byte
pieces and in single words, tile order forwards and backwards.  A lattice
stepped alone and one in a batch take different ones of these and must agree
bit for bit; masks that put walls at every distance from a tile's edge are held
to the FP64 oracle."""
import numpy as np
import pytest

from paper_1904_06881_gb300 import workloads as W

from helpers import gpu_from_workload, normwise, oracle_from_workload

pytestmark = pytest.mark.gpu

STEPS = 5
# Five steps in FP32: a density is a sum of up to 27 populations that four
# operations a step round by 6e-8 of themselves, 1.5e-6 of rho_l = 6.1 or 2.6e-7
# of rho_l - rho_g a step at worst; the force feeds a few times that back.
TOL = 1e-5


def _wl(lattice, nx, ny, nz, mask, wetting=W.WET_FORCE, seed=0, **params):
    rng = np.random.default_rng(seed)
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(np.float64)
    n = (nx, ny, nz)
    c = [0.43 * n[0] + 0.3, 0.52 * n[1] + 0.2, 0.47 * n[2] + 0.1 if nz > 1 else 0.0]
    R = 0.3 * min(k for k in n if k > 1)
    C2 = 0.5 * (1.0 - np.tanh((np.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) - R) / 2.0))
    C3 = rng.uniform(-1e-3, 1e-3, C2.shape)
    rho, phi = W.phase_fields(C2, C3)
    p = W.base_params(wetting=wetting, **params)
    if wetting == W.WET_FORCE:
        p["kw_rho"] = 0.05
    else:
        p["theta_deg"] = (70.0, 70.0, 90.0)
    return dict(name="variants", lattice=lattice, nx=nx, ny=ny, nz=nz, mask=mask, rho=rho, phi=phi, params=p)


def _mask(nx, ny, nz, kind):
    m = np.zeros((nz, ny, nx), np.uint8)
    if kind == "plane":
        if nz > 1:
            m[0] = 1
        else:
            m[:, 0] = 1
    elif kind == "random":
        rng = np.random.default_rng(nx * 1000 + ny)
        for _ in range(3):                      # small blocks, the periodic edges among their places
            o = [int(rng.integers(0, k)) for k in (nz, ny, nx)]
            idx = [np.arange(a, a + 3) % k for a, k in zip(o, (nz, ny, nx))]
            m[np.ix_(*idx) if nz > 1 else np.ix_([0], idx[1], idx[2])] = 1
    elif kind.startswith("block"):              # a block whose near face lies `d` nodes behind x = 32 or 16
        d = int(kind[5:])
        x0 = (32 if nz == 1 else 16) + d
        m[(slice(0, 3) if nz > 1 else 0), 2:5, x0:x0 + 3] = 1
    return m


@pytest.mark.parametrize("kind", ["plane", "random", "block0", "block1", "block2", "block3"])
@pytest.mark.parametrize("size", [(W.D2Q9, 67, 21, 1), (W.D2Q9, 64, 16, 1), (W.D3Q27, 35, 10, 9), (W.D3Q27, 32, 12, 8)])
def test_walls_at_every_distance_from_a_tile(size, kind):
    lattice, nx, ny, nz = size
    for wetting in (W.WET_FORCE, W.WET_GEOM_EXTRAP):
        wl = _wl(lattice, nx, ny, nz, _mask(nx, ny, nz, kind), wetting)
        g, o = gpu_from_workload(wl), oracle_from_workload(wl)
        g.step(STEPS)
        o.step(STEPS)
        e = normwise(g.fields(), o.fields(), o.derived, mask=wl["mask"])
        assert e["rho"] <= TOL and e["phi"] <= TOL and e["C"] <= TOL, (size, kind, wetting, e)


def _alone_and_batched(wls, steps=STEPS):
    from paper_1904_06881_gb300 import tlb

    alone = [gpu_from_workload(w) for w in wls]
    batched = [gpu_from_workload(w) for w in wls]
    for a in alone:
        a.step(steps)
    tlb.tlb_step_batch([b.h for b in batched], steps)
    for w, a, b in zip(wls, alone, batched):
        fa, fb = a.populations(), b.populations()
        fl = w["mask"].reshape(-1) == 0
        assert np.array_equal(fa[0][:, fl], fb[0][:, fl]) and np.array_equal(fa[1][:, fl], fb[1][:, fl]), \
            (w["nx"], w["ny"], w["nz"])
        a.close()
        b.close()


@pytest.mark.parametrize("nx,ny,nz", [(16, 8, 8), (17, 9, 7), (18, 7, 6), (19, 5, 9), (20, 6, 5), (33, 11, 10), (47, 6, 7),
                                      (6, 5, 5), (3, 3, 3)])
@pytest.mark.parametrize("fp16", [0, 1])
def test_staging_of_the_populations(nx, ny, nz, fp16):
    """Rows that start at every shift from a 16-byte boundary, and the array's last piece."""
    _alone_and_batched([_wl(W.D3Q27, nx, ny, nz, _mask(nx, ny, nz, "none"), g_fp16=fp16)])


@pytest.mark.parametrize("size", [(W.D2Q9, 1023, 255, 1), (W.D2Q9, 1025, 257, 1), (W.D3Q27, 130, 61, 33), (W.D3Q27, 96, 92, 88)])
def test_flags_as_parameters_and_from_memory(size):
    """1024 tiles and a few more; the last lattice is larger than the L2 cache and steps backwards."""
    _alone_and_batched([_wl(*size, _mask(*size[1:], "random"))], steps=3)


def test_a_new_mask_replaces_the_tile_flags():
    nx, ny, nz = 32, 12, 8
    a = _wl(W.D3Q27, nx, ny, nz, _mask(nx, ny, nz, "block2"))
    b = _wl(W.D3Q27, nx, ny, nz, _mask(nx, ny, nz, "plane"))
    lat, ref = gpu_from_workload(a), gpu_from_workload(b)
    lat.step(3)
    lat.set_solid(b["mask"])
    lat.init_fields(b["rho"], b["phi"])
    lat.step(STEPS)
    ref.step(STEPS)
    f, r = lat.fields(), ref.fields()
    assert np.array_equal(f["rho"], r["rho"]) and np.array_equal(f["phi"], r["phi"])
