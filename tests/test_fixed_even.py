"""Which elements the FP64 kernels keep in block fixed point (fe_fixed.cuh,
fe_fixed_prism.cuh), compiled for the CPU from the kernels' own headers with the tests
that the kernels use: elements in which a common unit would cost an entry of A^e more
than double's own cancellation are left to the double form, and ordinary ones are kept."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1504_01023_gb300 import meshgen
from test_fixed_algorithm import CSRC, PRISM_SHIM, SHIM, fixed, prism_fixed, prism_reference, reference, rel

EPS = [2.0 ** -p for p in (1, 3, 5, 7, 8, 9, 10, 20, 40)]


def _compile(d, name, src):
    path, out = str(d / (name + ".cpp")), str(d / (name + ".so"))
    with open(path, "w") as f:
        f.write(src)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    CSRC, path, "-o", out], check=True)
    return ctypes.CDLL(out)


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    """The shims of the algorithm's tests with the kernels' tests switched on."""
    d = tmp_path_factory.mktemp("even")
    tet = SHIM.replace("geometry(Arr{x + 12 * e})", "geometry(Arr{x + 12 * e}) && f.even_rows()")
    tet = tet.replace("        f.laplace(L + 16 * e);", "        ok[2 * e] = f.laplace(L + 16 * e);")
    tet = tet.replace("= four ?", "= f.even(cc) && (four ?").replace("b + 4 * e);\n    }", "b + 4 * e));\n    }")
    prism = PRISM_SHIM.replace("template exponents<KIND>(", "template exponents<KIND, true>(")
    prism = prism.replace("            P[l].template gamma", "            if (KIND) P[l].ok = P[l].ok && P[l].even_shape();\n"
                          "            P[l].template gamma")
    assert "even_rows" in tet and "= f.laplace" in tet and "f.even(cc)" in tet and "KIND, true" in prism and "even_shape" in prism
    return _compile(d, "tet", tet), _compile(d, "prism", prism)


def _diffusion(n, points, d):
    c = np.zeros((n, points, 20))
    for i in range(3):
        c[..., 5 + 5 * i] = d[i]
    c[..., 16] = 1.0
    return c


def _entry_errors(got, ref):
    """Largest relative error of an element's entries that are not zero."""
    ref = np.asarray(ref, dtype=np.longdouble)
    nz = ref != 0
    return np.where(nz, np.abs(got - ref) / np.where(nz, np.abs(ref), 1), 0).reshape(len(ref), -1).max(1).astype(float)


# Structured elements on a grid of 2^-3: double evaluates their entries almost exactly.
# An entry is at least 2^-9 of the largest where the element is kept (diagonal
# coefficients within 8 bits, one more for the geometry), its fixed-point error at most
# about 2^-56 of the largest: a relative error of 2^-47, with two bits to spare.
@pytest.mark.parametrize("four", [0, 1])
@pytest.mark.parametrize("eps", EPS)
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_axis_aligned_anisotropy_tets(libs, eps, axis, four):
    x = meshgen.tet_cube_mesh(8, 0.0)
    d = [eps] * 3
    d[axis] = 1.0
    c = _diffusion(len(x), 1, d)[:, 0]
    A, b, L, vol, ok = fixed(libs[0], x, c, four)
    kept = ok.all(1)
    assert ok[:, 0].all() and kept.all() == (eps >= 2.0 ** -7) and kept.any() == kept.all()
    if kept.any():
        assert _entry_errors(A, reference(x, c, four, np.longdouble)[0]).max() <= 2.0 ** -45


@pytest.mark.parametrize("pq", [0, 1])
@pytest.mark.parametrize("eps", EPS)
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_axis_aligned_anisotropy_prisms(libs, eps, axis, pq):
    x = meshgen.prism_slab_mesh(16, zjitter=0.0)
    d = [eps] * 3
    d[axis] = 1.0
    c = _diffusion(len(x), 6 if pq else 1, d)
    A, b, ok = prism_fixed(libs[1], x, c, 1, pq)
    assert ok.all() == (eps >= 2.0 ** -6) and ok.any() == ok.all()
    if ok.any():
        ref = prism_reference(x, c, 1, pq, np.longdouble)[0]
        # entries that cancel to rounding (of the rule's points) are zero
        ref = np.where(np.abs(ref) > 1e-15 * np.abs(ref).max(), ref, 0)
        A = np.where(ref == 0, 0, A)
        assert _entry_errors(A, ref).max() <= 2.0 ** -45


def test_ordinary_elements_are_kept(libs):
    """Jittered meshes with the benchmark's coefficients: a whole warp runs the double
    form for one element that is left, so at most one in 10,000 may be."""
    x = meshgen.tet_cube_mesh(24, seed=8)
    for four in (0, 1):
        A, b, L, vol, ok = fixed(libs[0], x, meshgen.generic_coefs(len(x), seed=9), four)
        assert ok.all(1).mean() >= 0.9999
    x = meshgen.prism_slab_mesh(100, seed=8)
    for pq in (0, 1):
        A, b, ok = prism_fixed(libs[1], x, meshgen.generic_coefs(len(x), 6 if pq else 1, seed=9).reshape(len(x), -1, 20), 1,
                               pq)
        assert ok.mean() >= 0.9999


def test_zero_coefficients_do_not_count(libs):
    """Elements without an operator or with diffusion along some axes only are kept."""
    x = meshgen.tet_cube_mesh(6, seed=4)
    p = meshgen.prism_slab_mesh(10, seed=4)
    for d in ([0, 0, 0], [1, 0, 0], [0, 2.0, 1.0], [-1.0, 1.0, 0]):
        c = _diffusion(len(x), 1, d)[:, 0]
        c[:, 0] = c[:, 1] = 1e-3
        A, b, L, vol, ok = fixed(libs[0], x, c, 1)
        assert ok.all()
        assert rel(A, reference(x, c, 1, np.longdouble)[0]).max() <= 1e-12
        c = _diffusion(len(p), 6, d)
        c[..., 0] = c[..., 1] = 1e-3
        A, b, ok = prism_fixed(libs[1], p, c, 1, 1)
        assert ok.all()
        assert rel(A, prism_reference(p, c, 1, 1, np.longdouble)[0]).max() <= 1e-12


def _stretch(rng, x, k):
    """Elements stretched k times along a direction of their own."""
    q = meshgen._haar_orthogonal(rng, len(x))
    m = np.einsum("nij,j,nkj->nik", q, np.array([1, 1, k]), q)
    return np.einsum("nvj,nij->nvi", x - x[:, :1], m) + x[:, :1]


def _tets(name, p, n=8000):
    """n tetrahedra with edges from vertex 0 of different lengths, by powers of two."""
    rng = np.random.default_rng(100 * p + sum(map(ord, name)))
    if name in ("stretch", "squash"):
        return _stretch(rng, meshgen.tet_cube_mesh(12, seed=3)[:n], 2.0 ** (p if name == "stretch" else -p))
    e = rng.uniform(-1, 1, (n, 3, 3))
    if name == "long":     # one edge along (1, 1, 1), off the axes
        e[:, 2] = 2.0 ** p / np.sqrt(3) * rng.uniform(1, 2, (n, 1)) + 0.5 * e[:, 2]
    else:
        e[:, 1 if name == "two_short" else 2:] *= 2.0 ** -p
    return np.concatenate([np.zeros((n, 1, 3)), e], 1) + rng.uniform(0, 1, (n, 1, 3))


def _points(v):
    """Median, 99% point and maximum: rms values of these families are those of a few
    nearly degenerate elements, in which either form may be the luckier."""
    return np.median(v), np.quantile(v, 0.99), v.max()


@pytest.mark.parametrize("name", ["long", "two_short", "one_short", "stretch", "squash"])
@pytest.mark.parametrize("p", [0, 1, 2, 3, 4, 6, 8])
def test_uneven_tets_no_further_than_double(libs, name, p):
    """What is kept of families of short and long edges is as near to the exact results as
    plain double evaluation, in the norm of A^e and b^e: the median no further, the 99%
    point within one bit. One edge 2^4 times the others is not kept."""
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision on this machine")
    x = _tets(name, p)
    c = meshgen.generic_coefs(len(x), seed=p)
    A, b, L, vol, ok = fixed(libs[0], x, c, 1)
    ref, dbl = reference(x, c, 1, np.longdouble), reference(x, c, 1, np.float64)
    if name == "long" and p >= 4:
        assert not ok.any()
    for got, d, r, kept in zip((A, b, L), dbl, ref, (ok[:, 1], ok[:, 1], ok[:, 0])):
        if kept.sum() >= 400:
            (mg, qg, _), (md, qd, _) = _points(rel(got, r)[kept]), _points(rel(d, r)[kept])
            assert mg <= md and qg <= 2 * qd


@pytest.mark.parametrize("pq", [0, 1])
@pytest.mark.parametrize("name", ["stretch", "squash", "shear", "flat", "tall"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
def test_uneven_prisms_no_further_than_double(libs, name, p, pq):
    """The same for generic prisms, within one bit throughout, the maximum too; flat and
    tall ones are kept whole."""
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision on this machine")
    rng = np.random.default_rng(7 * p + pq)
    x = meshgen.prism_slab_mesh(32, seed=5)
    if name in ("stretch", "squash"):
        x = _stretch(rng, x, 2.0 ** (p if name == "stretch" else -p))
    elif name == "shear":
        x = x + x[..., 2:] * np.array([2.0 ** p, 0, 0])
    else:
        x = x * np.array([1, 1, 2.0 ** (p if name == "tall" else -p)])
    c = meshgen.generic_coefs(len(x), 6 if pq else 1, seed=p).reshape(len(x), -1, 20)
    A, b, ok = prism_fixed(libs[1], x, c, 1, pq)
    if name in ("flat", "tall"):
        assert ok.mean() >= 0.999
    if ok.sum() >= 100:
        ref, dbl = prism_reference(x, c, 1, pq, np.longdouble), prism_reference(x, c, 1, pq, np.float64)
        for got, d, r in zip((A, b), dbl, ref):
            for eg, ed in zip(_points(rel(got, r)[ok]), _points(rel(d, r)[ok])):
                assert eg <= 2 * ed
