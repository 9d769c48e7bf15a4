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
    tet = SHIM.replace("= four ?", "= f.even(cc) && (four ?").replace("b + 4 * e);\n    }", "b + 4 * e));\n    }")
    prism = PRISM_SHIM.replace("template exponents<KIND>(", "template exponents<KIND, true>(")
    assert tet != SHIM and prism != PRISM_SHIM
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
