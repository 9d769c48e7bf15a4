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


# ---------------------------------------------------------------------------
# Prisms: both levels of an element in step, as the two threads of a pair run them
# ---------------------------------------------------------------------------
PRISM_SHIM = r"""
#include "fe_fixed_prism.cuh"
using namespace fe;
struct Arr { const double *p; double operator()(int j) const { return p[j]; } };
template <int KIND> static bool one(const double *x, const double *c, int pq, double *A, double *b) {
    PrismFx P[2];
    int64_t scratch[2][60];
    const int st = KIND ? 20 : 1, np = pq ? 3 : 1;
    const Arr C[2] = {{c}, {c + (pq ? 3 * st : 0)}};
    uint32_t b12 = 0, b3 = 0, d = 0;
    for (int l = 0; l < 2; ++l) {
        P[l].v = scratch[l];
        uint32_t u, w;
        P[l].begin(Arr{x}, l, u, w);
        b12 |= u;
        b3 |= w;
    }
    if (!P[0].ok) return false;
    for (int l = 0; l < 2; ++l) d |= P[l].set_a(b12, b3);
    for (int l = 0; l < 2; ++l) {
        P[l].set_det(d);
        P[l].template exponents<KIND>(C[l], np);
    }
    for (int j = 0; j < 6; ++j) P[0].En[j] = P[1].En[j] = fx_maxi(P[0].En[j], P[1].En[j]);
    for (int l = 0; l < 2; ++l) {
        P[l].template common_exponents<KIND>();
        P[l].template set_exponents<KIND>(C[l], np);
    }
    for (int t = 0; t < 3; ++t) {
        int T12[2], T3[2];
        for (int l = 0; l < 2; ++l) P[l].template products<KIND>(C[l], pq ? st : 0, t, T12[l], T3[l]);
        for (int l = 0; l < 2; ++l) {
            if (t == 0) P[l].set_products(fx_maxi(T12[0], T12[1]), fx_maxi(T3[0], T3[1]));
            P[l].template gamma<KIND>(t);
        }
    }
    for (int l = 0; l < 2; ++l) P[l].template sums<KIND>();
    if (!P[0].ok || !P[1].ok) return false;
    const int ta = fx_mini(P[0].lza, P[1].lza), tb = fx_mini(P[0].lzb, P[1].lzb);
    for (int l = 0; l < 2; ++l) P[l].template align<KIND>(ta, tb);
    for (int i = 0; i < 9; ++i) {
        int64_t X[2], Y[2], U[2], V[2];
        for (int l = 0; l < 2; ++l) P[l].blocks(l, i, X[l], Y[l], U[l], V[l]);
        const int64_t x = X[0] + X[1], y = Y[0] + Y[1], u = U[0] + U[1], v = V[0] + V[1];
        const int k = i / 3, kk = i % 3;
        A[6 * k + kk] = P[0].out_a(x + y);
        A[6 * (k + 3) + kk + 3] = P[0].out_a(x - y);
        A[6 * k + kk + 3] = P[0].out_a(u + v);
        A[6 * (k + 3) + kk] = P[0].out_a(u - v);
    }
    for (int k = 0; k < 3; ++k) {
        int64_t X[2], Y[2];
        for (int l = 0; l < 2; ++l) P[l].loads(l, k, X[l], Y[l]);
        b[k] = P[0].out_b(X[0] + X[1] + Y[0] + Y[1]);
        b[k + 3] = P[0].out_b(X[0] + X[1] - Y[0] - Y[1]);
    }
    return true;
}
extern "C" void fx_prism(long n, const double *x, const double *c, int kind, int pq, double *A, double *b, int *ok) {
    const int nc = (kind ? 20 : 1) * (pq ? 6 : 1);
    for (long e = 0; e < n; ++e)
        ok[e] = kind ? one<1>(x + 18 * e, c + nc * e, pq, A + 36 * e, b + 6 * e)
                     : one<0>(x + 18 * e, c + nc * e, pq, A + 36 * e, b + 6 * e);
}
"""


@pytest.fixture(scope="module")
def prism_lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxp")
    src, out = str(d / "fxp.cpp"), str(d / "fxp.so")
    with open(src, "w") as f:
        f.write(PRISM_SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    CSRC, src, "-o", out], check=True)
    return ctypes.CDLL(out)


def prism_fixed(lib, x, c, kind, pq):
    n = len(x)
    A, b, ok = np.zeros((n, 6, 6)), np.zeros((n, 6)), np.zeros(n, dtype=np.int32)
    x, c = np.ascontiguousarray(x), np.ascontiguousarray(c)
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, c, A, b, ok)]
    lib.fx_prism(ctypes.c_long(n), p[0], p[1], ctypes.c_int(kind), ctypes.c_int(pq), p[2], p[3], p[4])
    return A, b, ok.astype(bool)


def prism_reference(x, c, kind, pq, dt):
    """A, b by the six-point sum in precision dt; c [n, points, k]."""
    x, c = x.astype(dt), c.astype(dt)
    xe = x - x[:, :1]
    n = len(x)
    A, b = np.zeros((n, 6, 6), dtype=dt), np.zeros((n, 6), dtype=dt)
    dl = np.array([[-1, -1], [1, 0], [0, 1]], dtype=dt)
    for q in range(6):
        l, t = divmod(q, 3)
        z = (1 if l else -1) / np.sqrt(dt(3))
        zz = [(1 - z) / 2, (1 + z) / 2]
        lam = np.array([dt(2) / 3 if k == t else dt(1) / 6 for k in range(3)])
        ph = np.concatenate([lam * zz[0], lam * zz[1]])
        de = np.zeros((6, 3), dtype=dt)
        de[:3, :2], de[3:, :2], de[:3, 2], de[3:, 2] = dl * zz[0], dl * zz[1], -lam / 2, lam / 2
        J = np.einsum("nrd,rj->ndj", xe, de)
        cof = np.stack([np.cross(J[..., 1], J[..., 2]), np.cross(J[..., 2], J[..., 0]),
                        np.cross(J[..., 0], J[..., 1])], 1)
        det = (J[..., 0] * cof[:, 0]).sum(-1)
        g = np.einsum("rj,njd->nrd", de, cof) / det[:, None, None]
        vol = np.abs(det) / dt(6)
        cq = c[:, q if pq else 0]
        if kind == 0:
            A += vol[:, None, None] * np.einsum("nri,nsi->nrs", g, g)
            b += (vol * cq[:, 0])[:, None] * ph
        else:
            P = np.concatenate([np.broadcast_to(ph[None, :, None], (n, 6, 1)), g], 2)
            A += vol[:, None, None] * np.einsum("nri,nij,nsj->nrs", P, cq[:, :16].reshape(-1, 4, 4), P)
            b += vol[:, None] * np.einsum("nri,ni->nr", P, cq[:, 16:])
    return A, b


def prism_family(name, kind, pq, n=1500):
    rng = np.random.default_rng(sum(map(ord, name)))
    h = {"fine": 1e-3, "large": 1e2}.get(name, 1e-2)
    hz = h * {"thin": 0.1, "tall": 50.0}.get(name, 1.0)
    base = np.array([[0, 0], [1, 0], [1, 1.0]])
    x = np.empty((n, 6, 3))
    x[:, :, :2] = np.concatenate([base, base])[None] * h + rng.uniform(0, 1, (n, 1, 2)) * (h if name == "large" else 1)
    if name == "skewed":
        x[:, :, :2] += 0.2 * h * rng.uniform(-1, 1, (n, 6, 2))
    x[:, :, 2] = np.repeat([0.0, hz], 3) + 0.1 * hz * rng.uniform(-1, 1, (n, 6))
    if name == "inverted":
        x[:, :, 2] *= -1
    nq = 6 if pq else 1
    if kind == 0:
        return x, rng.uniform(-1, 1, (n, nq, 1))
    c = rng.uniform(-1, 1, (n, nq, 20))
    for i in range(3):
        for j in range(3):
            c[..., 4 * i + j + 5] = (4.9 if i == j else 2) * c[..., 4 * i + j + 5] + (5.0 if i == j else 0.0)
    if name == "mass":
        c[..., 1:16] = 0
    if name == "no_load":
        c[..., 16:] = 0
    return x, c


@pytest.mark.parametrize("kind,pq", [(1, 1), (1, 0), (0, 1), (0, 0)])
@pytest.mark.parametrize("name", ["regular", "fine", "large", "thin", "tall", "skewed", "inverted", "mass", "no_load"])
def test_prism_fixed_point_no_further_than_double(prism_lib, name, kind, pq):
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision on this machine")
    x, c = prism_family(name, kind, pq)
    A, b, ok = prism_fixed(prism_lib, x, c, kind, pq)
    assert ok.mean() > 0.999
    ref, dbl = prism_reference(x, c, kind, pq, np.longdouble), prism_reference(x, c, kind, pq, np.float64)
    for got, d, r in zip((A, b), dbl, ref):
        eg, ed = rel(got, r)[ok], rel(d, r)[ok]
        assert eg.max() <= 1e-12
        assert np.sqrt((eg ** 2).mean()) <= np.sqrt((ed ** 2).mean())


def test_prism_out_of_window_elements_are_left(prism_lib):
    x, c = prism_family("regular", 1, 1, 16)
    x[0, 3:] = x[0, :3]                                # flat
    x[1] *= 2.0 ** 300
    x[2] = (x[2] - x[2, 0]) * 2.0 ** -300
    x[3, 4, 1] = np.inf
    x[4, 4, 1] = np.nan
    x[5, 3:, 2] = x[5, :3, 2] + 1e-2 * np.array([1.0, 1.0, -0.5])      # det near 0 at a point
    x[9, 3:, 2] = x[9, :3, 2] + 1e-2 * np.array([1.0, 1.0, -1.0])      # det of both signs: taken
    c[6, 3, 6] = np.inf
    c[7, 1, 0] = np.nan
    c[8, 5, 18] = np.nan
    A, b, ok = prism_fixed(prism_lib, x, c, 1, 1)
    assert not ok[:9].any() and ok[9:].all()
    Ar, br = prism_reference(x[9:], c[9:], 1, 1, np.longdouble)
    assert rel(A[9:], Ar).max() <= 1e-12 and rel(b[9:], br).max() <= 1e-12


def test_prism_largest_operands_do_not_overflow(prism_lib):
    """Significands and limbs at their extremes in every coordinate difference and coefficient."""
    rng = np.random.default_rng(4)
    n = 4000
    top = 2.0 - 2.0 ** -52
    vals = np.array([top, -top, 1.0 + 2.0 ** -28, -1.0 - 2.0 ** -28, 1.0, -1.0, 0.0])
    x = np.zeros((n, 6, 3))
    x[:, 1:] = vals[rng.integers(0, 7, (n, 5, 3))]
    for kind in (0, 1):
        c = vals[rng.integers(0, 6, (n, 6, 20 if kind else 1))]
        A, b, ok = prism_fixed(prism_lib, x, c, kind, 1)
        Ar, br = prism_reference(x[ok], c[ok], kind, 1, np.longdouble)
        big = np.sqrt((Ar.astype(np.float64) ** 2).reshape(len(Ar), -1).sum(1)) > 1e-3
        assert big.sum() > 20
        assert rel(A[ok], Ar)[big].max() <= 1e-12
