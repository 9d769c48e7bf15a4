"""Block fixed-point contractions of the FP64 form (fe_fixed.cuh), compiled for
the CPU from the kernels' own header and compared with the same integrals in
extended precision: on every family of elements and coefficients the fixed-point
results must be no further from them than the plain double evaluation (rms over
the family), and within the FP64 form's tolerance (1e-12 per element, relative
Frobenius norm); elements outside the windows must be left to the double form."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_01023_gb300", "csrc")
SHIM = r"""
#include "fe_fixed.cuh"
using namespace fe;
struct Arr { const double *p; double operator()(int j) const { return p[j]; } };
extern "C" void fx_tet(long n, const double *x, const double *c, int four, double *A, double *b, double *L,
                       double *vol, int *ok) {
    for (long e = 0; e < n; ++e) {
        TetFx f;
        ok[2 * e] = f.geometry(Arr{x + 12 * e});
        ok[2 * e + 1] = 0;
        if (!ok[2 * e]) continue;
        f.laplace(L + 16 * e);
        vol[e] = f.volume();
        const Arr cc{c + 20 * e};
        ok[2 * e + 1] = four ? f.generic<true>(cc, A + 16 * e, b + 4 * e) : f.generic<false>(cc, A + 16 * e, b + 4 * e);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, out = str(d / "fx.cpp"), str(d / "fx.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    CSRC, src, "-o", out], check=True)
    return ctypes.CDLL(out)


def fixed(lib, x, c, four):
    n = len(x)
    A, b, L = np.zeros((n, 4, 4)), np.zeros((n, 4)), np.zeros((n, 4, 4))
    vol, ok = np.zeros(n), np.zeros((n, 2), dtype=np.int32)
    x, c = np.ascontiguousarray(x), np.ascontiguousarray(c)
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, c, A, b, L, vol, ok)]
    lib.fx_tet(ctypes.c_long(n), p[0], p[1], ctypes.c_int(four), p[2], p[3], p[4], p[5], p[6])
    return A, b, L, vol, ok.astype(bool)


def reference(x, c, four, dt):
    """A, b, Laplace A in precision dt, by the closed reference sums."""
    x, c = x.astype(dt), c.astype(dt)
    e = x[:, 1:] - x[:, :1]
    a = np.stack([np.cross(e[:, 1], e[:, 2]), np.cross(e[:, 2], e[:, 0]), np.cross(e[:, 0], e[:, 1])], 1)
    det = (e[:, 0] * a[:, 0]).sum(-1)
    a = np.concatenate([-a.sum(1, keepdims=True), a], 1)
    V, sg, W = np.abs(det), np.sign(det), dt(1) / dt(6)
    C = c[:, :16].reshape(-1, 4, 4)
    K = np.einsum("nri,nij,nsj->nrs", a, C[:, 1:, 1:], a)
    cr, cs = np.einsum("nri,ni->nr", a, C[:, 1:, 0]), np.einsum("nri,ni->nr", a, C[:, 0, 1:])
    M = W / 20 * (1 + np.eye(4, dtype=dt)) if four else np.full((4, 4), W / 16, dtype=dt)
    A = ((W / V)[:, None, None] * K + (sg * W / 4)[:, None, None] * (cr[:, :, None] + cs[:, None, :]) +
         (V * C[:, 0, 0])[:, None, None] * M)
    b = sg[:, None] * W * np.einsum("nri,ni->nr", a, c[:, 17:]) + (V * c[:, 16] * W / 4)[:, None]
    return A, b, (W / V)[:, None, None] * np.einsum("nri,nsi->nrs", a, a)


def family(name, n=4000):
    rng = np.random.default_rng(sum(map(ord, name)))
    base = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], [1, 1, 1.0]])
    h = {"fine": 1e-4, "large": 1e3}.get(name, 1e-2)
    if name == "scales":
        h = np.exp2(rng.uniform(-60, 60, (n, 1, 1)))
    jit = 0.0 if name == "structured" else 0.2
    o = rng.uniform(0, 1, (n, 1, 3)) * (h if name in ("large", "scales") else 1.0)
    x = o + h * (base + jit * rng.uniform(-1, 1, (n, 4, 3)))
    if name == "flat":
        x[:, :, 2] = o[:, :, 2] + 0.05 * (x[:, :, 2] - o[:, :, 2])
    if name == "thin":
        x[:, :, 2] = o[:, :, 2] + 1e-3 * (x[:, :, 2] - o[:, :, 2])
    if name == "long":
        x[:, :, 1:] = o[:, :, 1:] + 1e-3 * (x[:, :, 1:] - o[:, :, 1:])
    if name == "slivers":
        t = np.exp(rng.uniform(np.log(2e-3), np.log(2e-2), (n, 1)))
        m = x[:, :3].mean(1)
        x[:, 3] = m + t * (x[:, 3] - m)
    if name == "inverted":
        x[:, [1, 2]] = x[:, [2, 1]]
    c = rng.uniform(-1, 1, (n, 20))
    for i in range(3):
        for j in range(3):
            c[:, 4 * i + j + 5] = 2 * c[:, 4 * i + j + 5] + (5.0 if i == j else 0.0)
    if name == "mass":
        c[:, 1:16] = 0
    if name == "advection":
        for i in range(3):
            c[:, 4 * i + 5:4 * i + 8] = 0
        c[:, 0] = 0
    if name == "wild":
        c = np.ldexp(c, rng.integers(-20, 20, c.shape))
    if name == "no_load":
        c[:, 16:] = 0
    if name == "no_operator":
        c[:, :16] = 0
    return x, c


def rel(v, r):
    d = np.sqrt(((v - r).astype(np.float64) ** 2).reshape(len(v), -1).sum(1))
    m = np.sqrt((r.astype(np.float64) ** 2).reshape(len(v), -1).sum(1))
    return np.where(m > 0, d / np.where(m > 0, m, 1), d)


@pytest.mark.parametrize("four", [0, 1])
@pytest.mark.parametrize("name", ["regular", "structured", "fine", "large", "scales", "flat", "thin", "long", "slivers", "inverted",
                                  "mass", "advection", "wild", "no_load", "no_operator"])
def test_fixed_point_no_further_than_double(lib, name, four):
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision on this machine")
    x, c = family(name)
    A, b, L, vol, ok = fixed(lib, x, c, four)
    assert ok.all()
    ref, dbl = reference(x, c, four, np.longdouble), reference(x, c, four, np.float64)
    for got, d, r in zip((A, b, L), dbl, ref):
        eg, ed = rel(got, r), rel(d, r)
        assert eg.max() <= 1e-12
        assert np.sqrt((eg ** 2).mean()) <= np.sqrt((ed ** 2).mean())
    r0 = np.abs(np.linalg.det((x[:, 1:] - x[:, :1]).astype(np.float64)))
    assert np.abs(vol / r0 - 1).max() <= 1e-12


def test_out_of_window_elements_are_left(lib):
    x, c = family("regular", 16)
    x[0, 1] = x[0, 0]                                  # degenerate
    x[1, 3] = x[1, :3].mean(0)                         # flat to rounding
    x[2] *= 2.0 ** 300                                 # edges above the window
    x[3] = (x[3] - x[3, 0]) * 2.0 ** -300              # below it
    x[4, 2, 1] = np.inf
    x[5, 2, 1] = np.nan
    s = np.array([0, 1, 2, 3.0])[:, None] * 1e-2
    x[6] = s + 1e-5 * (x[6] - x[6, :1])                # a needle along (1, 1, 1)
    c[7, 6] = np.inf
    c[8, 0] = np.nan
    c[9, 18] = np.nan
    c[10, :16] *= 2.0 ** 700
    c[11, 16:] *= 2.0 ** -750
    A, b, L, vol, ok = fixed(lib, x, c, 1)
    assert not ok[:7, 0].any() and ok[7:, 0].all()
    assert not ok[7:12, 1].any() and ok[12:, 1].all()


def test_largest_operands_do_not_overflow(lib):
    """Significands and limbs at their extremes: every coordinate difference and
    coefficient one ulp below a power of two, or whose low limb is -2^31."""
    rng = np.random.default_rng(3)
    n = 2000
    top = 2.0 - 2.0 ** -52
    half_limb = 1.0 + 2.0 ** -29                       # low 32 bits of the 61-bit integer exactly 2^31
    vals = np.array([top, -top, half_limb, -half_limb, 1.0, -1.0, 0.0])
    e = vals[rng.integers(0, 7, (n, 3, 3))]
    x = np.concatenate([np.zeros((n, 1, 3)), e], 1)
    c = vals[rng.integers(0, 6, (n, 20))]
    keep = np.abs(np.linalg.det(e)) > 1e-3
    x, c = x[keep], c[keep]
    for four in (0, 1):
        A, b, L, vol, ok = fixed(lib, x, c, four)
        ref = reference(x, c, four, np.longdouble)
        for got, r, m in zip((A, b, L), ref, (ok.all(1), ok.all(1), ok[:, 0])):
            big = np.sqrt((r.astype(np.float64) ** 2).reshape(len(r), -1).sum(1)) > 1e-6
            assert (m & big).sum() > 100
            assert rel(got, r)[m & big].max() <= 1e-12
