"""The kernels' roots of the entropic equation against the exact one: the short
form (two terms, up to max|x| = ALPHA_SHORT_MAX) is as exact in FP32 as the full
series.  The functions are compiled for the host from the kernels' header."""
import ctypes
import itertools
import os
import subprocess

import numpy as np
import pytest

from paper_1904_06881_gb300 import build as B

SOURCE = r"""
#include "tlb_device.cuh"
extern "C" float short_max() { return tlb::ALPHA_SHORT_MAX; }
extern "C" void roots(int n, const float *a, float *s, float *l)
{
    for (int k = 0; k < n; ++k, a += 6) {
        s[k] = tlb::alpha_short(a[0], a[1], a[2]);
        l[k] = tlb::alpha_series(a[0], a[1], a[2], a[3], a[4], a[5]);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("root")
    src, so = os.path.join(d, "root.cu"), os.path.join(d, "libroot.so")
    with open(src, "w") as fh:
        fh.write(SOURCE)
    subprocess.check_call([B._nvcc()] + B.ARCH + ["-O2", "-std=c++17", "-diag-suppress", "177", "-Xcompiler",
                                                  "-fPIC,-ffp-contract=off", "-I", B.CSRC, "-I",
                                                  os.path.join(B.ROOT, "include"), "-shared", "-o", so, src])
    L = ctypes.CDLL(so)
    L.short_max.restype = ctypes.c_float
    return L


def _states(D, n, X, skew, rng):
    """Mirror states f' and x = D/f' with max|x| = X: D = f^eq - f' without mass and momentum."""
    c = np.array(list(itertools.product((0, 1, -1), repeat=D)))
    u = rng.uniform(-0.1, 0.1, (n, D))
    s = np.sqrt(1 + 3 * u * u)
    A, Bf = 2 - s, (2 * u + s) / (1 - u)
    feq = np.ones((n, len(c)))
    for a in range(D):
        feq *= np.where(c[:, a] == 0, 2 / 3 * A[:, a:a + 1], 1 / 6 * A[:, a:a + 1] * Bf[:, a:a + 1] ** c[:, a])
    y = -rng.random(feq.shape) ** 6 if skew else rng.standard_normal(feq.shape)
    M = np.concatenate([np.ones((1, len(c))), c.T])
    G = np.einsum("ai,ni,bi->nab", M, feq, M)
    k = np.linalg.solve(G, np.einsum("ai,ni->na", M, feq * y)[..., None])[..., 0]
    y = y - np.einsum("na,ai->ni", k, M)                       # D = f^eq y
    j = np.abs(y).argmax(1)
    top = y[np.arange(n), j]
    y *= (X / (1 + np.sign(top) * X) / np.abs(top))[:, None]   # x = y / (1 - y)
    f = (feq * (1 - y)).astype(np.longdouble)
    return f, (feq * y).astype(np.longdouble) / f


def _exact(f, x):
    L, a = np.log1p(x), np.full(len(f), 2, np.longdouble)
    for _ in range(8):                                         # Newton's method from 2, off by max|x|
        y = a[:, None] * x
        ph = sum(((-1) ** k) * y ** k / np.longdouble(k * (k - 1)) for k in range(2, 12))
        a = a - (f * (ph - y * L)).sum(1) / (f * x * (np.log1p(y) - L)).sum(1)
    return a


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("skew", [False, True])
@pytest.mark.parametrize("part", [1.0, 0.5])
def test_short_form_is_as_exact_as_the_series(lib, D, skew, part):
    n, X = 3000, part * lib.short_max()
    f, x = _states(D, n, X, skew, np.random.default_rng(7 * D + skew))
    assert X * (1 - 1e-6) <= np.abs(x).max() <= X * (1 + 3 * X)
    exact = _exact(f, x)
    f32, x32 = f.astype(np.float32), x.astype(np.float32)
    t, a = f32 * x32 * x32, np.empty((n, 6), np.float32)
    for k in range(6):
        a[:, k] = t.sum(1, dtype=np.float32)
        t = t * x32
    s, l = np.empty(n, np.float32), np.empty(n, np.float32)
    P = lambda v: v.ctypes.data_as(ctypes.POINTER(ctypes.c_float))
    lib.roots(n, P(a), P(s), P(l))
    es, el = np.abs(s - exact), np.abs(l - exact)
    # alpha < 4: half a unit in its last place, the terms' own roundings (1e-7 of
    # |alpha - 2| <= 0.4 max|x|) and what the short form leaves out, below 3.3e-9
    assert es.max() <= 2.0 ** -23 + 4e-8 * X + 3.3e-9, es.max()
    rms = lambda e: float(np.sqrt(np.mean(e * e)))
    assert rms(es) <= 1.01 * rms(el), (rms(es), rms(el))
