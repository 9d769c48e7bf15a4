"""Plane-major results inside larger planes (a pitch above the number of elements, as of a
part of a longer set): what follows each plane's elements is left as it was, whatever unit
of 16 bytes the last tile ends in, and the results are those of the oracle."""
import numpy as np
import pytest
import torch

from helpers import TOL, make_inputs, max_errors, run_oracle, to_device_inputs
from paper_1504_01023_gb300 import api, build, meshgen

pytestmark = pytest.mark.gpu
CASES = [(api.TET, api.GENERIC, api.QUAD_TET4, 0), (api.TET, api.POISSON, api.QUAD_TET1, 0),
         (api.PRISM, api.GENERIC, api.QUAD_PRISM6, 1), (api.PRISM, api.POISSON, api.QUAD_PRISM6, 1)]


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = api.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("et,kind,quad,cpq", CASES)
@pytest.mark.parametrize("prec", [api.FP64, api.FP32_MIXED, api.FP64_DW])
@pytest.mark.parametrize("layout", [api.SOA, api.AOS])
@pytest.mark.parametrize("n,pitch", [(1, 4), (253, 256), (254, 256), (255, 256), (257, 260), (512, 516), (1001, 1004)])
def test_following_values_are_kept(ctx, et, kind, quad, cpq, prec, layout, n, pitch):
    mesh = (meshgen.tet_cube_mesh(6, seed=5) if et == api.TET else meshgen.prism_slab_mesh(24, seed=5))[:n]
    mesh, c = make_inputs(et, kind, quad, cpq, seed=7, mesh=mesh)
    X, C, c_used = to_device_inputs(et, mesh, c, prec, layout)
    ns, dt = api.NS[et], torch.float32 if prec == api.FP32_MIXED else torch.float64
    if layout == api.SOA:      # inputs inside larger planes too
        def wide(v):
            w = torch.full((v.shape[0], pitch), float("nan"), dtype=v.dtype, device="cuda")
            w[:, :n] = v
            return w[:, :n]
        X, C = wide(X), wide(C)
    ref = run_oracle(et, kind, quad, cpq, mesh, c_used)[:2]
    for packed in ((False, True) if kind == api.POISSON else (False,)):
        na = ns * (ns + 1) // 2 if packed else ns * ns
        A, b = (torch.full((k, pitch), 77.0, dtype=dt, device="cuda") for k in (na, ns))
        flags = torch.full((n + 8,), 99, dtype=torch.uint8, device="cuda")
        ctx.integrate(et, X, C, kind, quad, api.PER_QPOINT if cpq else api.PER_ELEMENT, prec, layout, api.SOA,
                      out=(A[:, :n], b[:, :n], flags[:n]), packed=packed)
        ctx.sync()
        assert (A[:, n:] == 77).all() and (b[:, n:] == 77).all() and (flags[n:] == 99).all()
        An = A[:, :n].double().cpu().numpy().T
        if packed:
            iu, full = np.triu_indices(ns), np.zeros((n, ns, ns))
            full[:, iu[0], iu[1]] = An
            full[:, iu[1], iu[0]] = An
            An = full
        ea, eb = max_errors(An.reshape(n, ns, ns), b[:, :n].double().cpu().numpy().T, *ref)
        assert ea <= TOL[prec] and eb <= TOL[prec]
