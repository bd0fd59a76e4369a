"""The ghost value behind one fluid-facing direction (Sec. IV.A-B), compiled for
the host from the kernels' header: its last multiply-add carries one rounding,
so that it is the nearest FP32 value to what its operands give, and the local
beta of per-component viscosities likewise."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1904_06881_gb300 import build as B

SOURCE = r"""
#include "tlb_device.cuh"
struct Plane {                             // nodes of a wall-parallel plane, (rho, phi) of node (x, y)
    const float *r, *p;
    int nx;
    bool get(int x, int y, int z, float2 &m) const
    {
        m = make_float2(r[x + nx * z], p[x + nx * z]);
        (void)y;
        return true;
    }
};
static tlb::DevParams params(int wetting, float cot)
{
    tlb::DevParams q = {};
    q.rho_l = 6.0f;
    q.rho_g = 0.4f;
    q.chi = 5.0f;
    q.inv_chi = 0.2f;
    q.inv_rgl = 1.0f / (0.4f - 6.0f);
    q.wetting = wetting;
    for (int k = 0; k < 3; ++k) q.cot[k] = cot;
    q.nu_on = 1;
    q.nu[0] = 0.12f, q.nu[1] = 0.17f, q.nu[2] = 0.25f;
    return q;
}
// nodes 1 .. nx - 2 of `rows` rows of nx nodes, the wall normal along y
extern "C" void ghosts(int D, int wetting, float cot, const float *r, const float *p, int nx, int rows, float *gr, float *gp)
{
    const tlb::DevParams q = params(wetting, cot);
    const Plane a{r, p, nx};
    for (int z = D == 3; z < rows - (D == 3); ++z)
        for (int x = 3; x < nx - 3; ++x) {
            const float2 m = make_float2(r[x + nx * z], p[x + nx * z]);
            float &u = gr[x + nx * z], &v = gp[x + nx * z];
            if (D == 2) tlb::ghost_axis<2>(q, a, x, 0, z, 1, m, u, v);
            else tlb::ghost_axis<3>(q, a, x, 0, z, 1, m, u, v);
        }
}
extern "C" void betas(int n, const float *r, const float *p, float *b)
{
    const tlb::DevParams q = params(0, 0.f);
    for (int k = 0; k < n; ++k) b[k] = tlb::local_beta(q, r[k], p[k]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("ghost")
    src, so = os.path.join(d, "ghost.cu"), os.path.join(d, "libghost.so")
    with open(src, "w") as fh:
        fh.write(SOURCE)
    subprocess.check_call([B._nvcc()] + B.ARCH + ["-O2", "-std=c++17", "-diag-suppress", "177", "-Xcompiler",
                                                  "-fPIC,-ffp-contract=off", "-I", B.CSRC, "-I",
                                                  os.path.join(B.ROOT, "include"), "-shared", "-o", so, src])
    return ctypes.CDLL(so)


F = np.float32
P = lambda v: v.ctypes.data_as(ctypes.POINTER(ctypes.c_float))


def _fields(rows, nx, seed):
    rng = np.random.default_rng(seed)
    r = (rng.uniform(0.4, 6.0, (rows, nx))).astype(F)
    return r, rng.uniform(-4.0, 4.0, (rows, nx)).astype(F)


def _fma(a, b, c):
    """a b + c rounded once (the product of two FP32 values is exact in FP64; the sum's own
    FP64 rounding moves the result for one pair in 2^29 at most)."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


@pytest.mark.parametrize("cot", [0.577, -0.364, 1.7])
def test_extrapolated_ghost_is_rounded_once(lib, cot):
    rows, nx = 40, 300
    r, p = _fields(rows, nx, 3)
    gr, gp = np.zeros_like(r), np.zeros_like(p)
    lib.ghosts(2, 1, ctypes.c_float(cot), P(r), P(p), nx, rows, P(gr), P(gp))
    dr, dp = F(0.5) * (r[:, 4:-2] - r[:, 2:-4]), F(0.5) * (p[:, 4:-2] - p[:, 2:-4])
    n = np.abs(dr)                             # in two dimensions the norm is the difference's size
    i23 = n < F(0.01) * F(F(6.0) - F(0.4)) * F(0.2) * np.abs(dp)
    t = np.sign(np.where(i23, dp, dr)).astype(F)
    for g, m, d in ((gr, r, dr), (gp, p, dp)):
        assert np.array_equal(g[:, 3:-3], _fma(np.full_like(d, cot), d * t, m[:, 3:-3]))


def test_interpolated_ghost_is_rounded_once(lib):
    rows, nx, cot = 40, 300, F(0.577)
    r, p = _fields(rows, nx, 4)
    gr, gp = np.zeros_like(r), np.zeros_like(p)
    lib.ghosts(2, 2, ctypes.c_float(cot), P(r), P(p), nx, rows, P(gr), P(gp))
    dr, dp = F(0.5) * (r[:, 4:-2] - r[:, 2:-4]), F(0.5) * (p[:, 4:-2] - p[:, 2:-4])
    i23 = np.abs(dr) < F(0.01) * F(F(6.0) - F(0.4)) * F(0.2) * np.abs(dp)
    l = cot * np.sign(np.where(i23, dp, dr)).astype(F)
    l0 = np.floor(l).astype(int)
    x = np.arange(3, nx - 3)[None, :] + l0
    for g, m in ((gr, r), (gp, p)):
        v0, v1 = np.take_along_axis(m, x, 1), np.take_along_axis(m, x + 1, 1)
        assert np.array_equal(g[:, 3:-3], _fma(l - l0.astype(F), v1 - v0, v0))


def test_three_dimensional_ghost(lib):
    """The extrapolation's sum over both in-plane axes: nearer to the FP64 value than two
    roundings of the norm, the unit vector and the products leave."""
    rows, nx, cot = 40, 300, F(0.577)
    r, p = _fields(rows, nx, 5)
    gr, gp = np.zeros_like(r), np.zeros_like(p)
    lib.ghosts(3, 1, ctypes.c_float(cot), P(r), P(p), nx, rows, P(gr), P(gp))
    D = np.float64
    cut = lambda m, dz, dx: m[1 + dz:rows - 1 + dz, 3 + dx:nx - 3 + dx].astype(D)
    diff = lambda m: (0.5 * (cut(m, 0, 1) - cut(m, 0, -1)), 0.5 * (cut(m, 1, 0) - cut(m, -1, 0)))
    (rx, rz), (px, pz) = diff(r), diff(p)
    nr, npp = np.hypot(rx, rz), np.hypot(px, pz)
    i23 = nr < 0.01 * 5.6 * 0.2 * npp
    tx, tz = np.where(i23, px, rx) / np.where(i23, npp, nr), np.where(i23, pz, rz) / np.where(i23, npp, nr)
    for g, m, a, b in ((gr, r, rx, rz), (gp, p, px, pz)):
        e = np.abs(cut(g, 0, 0) - (cut(m, 0, 0) + D(cot) * (a * tx + b * tz)))
        assert e.max() <= 2.0 ** -24 * (np.abs(cut(g, 0, 0)).max() + 6 * np.hypot(a, b).max())


def test_local_beta(lib):
    r, p = _fields(20, 500, 6)
    b = np.zeros_like(r)
    lib.betas(r.size, P(r), P(p), P(b))
    C1 = (r - F(6.0)) * F(F(1.0) / (F(0.4) - F(6.0)))
    C2, C3 = (F(0.5) * (_fma(s * p, np.full_like(p, 0.2), np.ones_like(p)) - C1) for s in (F(1), F(-1)))
    c1, c2, c3 = (np.clip(c, F(0), F(1)) for c in (C1, C2, C3))
    full = lambda v: np.full_like(p, v)
    nu = _fma(c1, full(0.12), _fma(c2, full(0.17), c3 * F(0.25))) / (c1 + c2 + c3)
    assert np.array_equal(b, F(1.0) / _fma(full(6.0), nu, full(1.0)))
