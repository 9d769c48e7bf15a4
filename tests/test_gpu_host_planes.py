"""Plane-major sets in pinned host memory whose forms take tiles moved by tensor copies
there (on the device they run straight from and to the planes), against the oracle: sizes
around a tile of 256 elements, planes that tensor copies can and cannot take, full and
packed outputs; nothing around the results is written."""
import numpy as np
import pytest
import torch

from helpers import TOL, make_inputs, max_errors, run_oracle
from paper_1504_01023_gb300 import api, build, meshgen

pytestmark = pytest.mark.gpu
CASES = [(api.TET, api.GENERIC, api.QUAD_TET4, 0, api.FP64), (api.TET, api.GENERIC, api.QUAD_TET1, 0, api.FP64),
         (api.TET, api.GENERIC, api.QUAD_TET4, 1, api.FP64), (api.TET, api.GENERIC, api.QUAD_TET4, 0, api.FP32_MIXED),
         (api.TET, api.GENERIC, api.QUAD_TET1, 1, api.FP32_MIXED), (api.TET, api.POISSON, api.QUAD_TET1, 0, api.FP64),
         (api.PRISM, api.POISSON, api.QUAD_PRISM6, 0, api.FP32_MIXED),
         (api.PRISM, api.POISSON, api.QUAD_PRISM6, 1, api.FP32_MIXED),
         (api.PRISM, api.GENERIC, api.QUAD_PRISM6, 0, api.FP32_MIXED)]


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _planes(k, n, pitch, dt):
    """[k, n] pinned planes `pitch` values apart, in a buffer of 77s."""
    buf = torch.full((k * pitch + 8,), 77.0, dtype=dt).pin_memory()
    return buf, buf[:k * pitch].view(k, pitch)[:, :n]


@pytest.mark.parametrize("et,kind,quad,cpq,prec", CASES)
@pytest.mark.parametrize("n,pitch", [(1, 1), (33, 33), (255, 256), (256, 256), (257, 260), (1001, 1001), (5000, 5000)])
def test_against_the_oracle(ctx, et, kind, quad, cpq, prec, n, pitch):
    mesh = (meshgen.tet_cube_mesh(10, seed=5) if et == api.TET else meshgen.prism_slab_mesh(50, seed=5))[:n].copy()
    if et == api.TET and prec == api.FP32_MIXED and n > 100:
        meshgen.make_slivers(mesh, 0.05, seed=6)
    mesh, c = make_inputs(et, kind, quad, cpq, seed=7, mesh=mesh)
    ns, cdt = api.NS[et], torch.float32 if prec == api.FP32_MIXED else torch.float64
    c = c.astype(np.float32 if prec == api.FP32_MIXED else np.float64)
    _, X = _planes(3 * ns, n, pitch, torch.float64)
    X.copy_(torch.from_numpy(mesh.reshape(n, -1).T.copy()))
    cc = c.reshape(n, -1)
    _, C = _planes(cc.shape[1], n, pitch, cdt)
    C.copy_(torch.from_numpy(cc.T.copy()))
    Ao, bo = run_oracle(et, kind, quad, cpq, mesh, c.astype(np.float64))[:2]
    for packed in ((False, True) if kind == api.POISSON else (False,)):
        na = ns * (ns + 1) // 2 if packed else ns * ns
        (ka, A), (kb, b) = _planes(na, n, pitch, cdt), _planes(ns, n, pitch, cdt)
        flags = torch.full((n + 8,), 99, dtype=torch.uint8).pin_memory()
        ctx.integrate(et, X, C, kind, quad, api.PER_QPOINT if cpq else api.PER_ELEMENT, prec, api.SOA, api.SOA,
                      out=(A, b, flags[:n]), packed=packed)
        An = A.numpy().T.astype(np.float64)
        if packed:
            iu, full = np.triu_indices(ns), np.zeros((n, ns, ns))
            full[:, iu[0], iu[1]] = An
            full[:, iu[1], iu[0]] = An
            An = full
        ea, eb = max_errors(An.reshape(n, ns, ns), b.numpy().T.astype(np.float64), Ao, bo)
        assert ea <= TOL[prec] and eb <= TOL[prec]
        assert (flags[:n] != 99).all() and (flags[n:] == 99).all()
        for k, v in ((ka, A), (kb, b)):
            pad = k[:v.shape[0] * pitch].view(-1, pitch)[:, n:]
            assert (pad == 77).all() and (k[v.shape[0] * pitch:] == 77).all()
