"""Elements that are left to the double form for their anisotropic diffusion, in FP64 on
every route of the kernels, mixed with ordinary ones in a warp. Tetrahedra: the largest
relative errors of an entry of A^e (99% point over the elements) within four times those
of the plain double evaluation: rounding orders differ, and the entries of vertex 0 come
from the sums of three others. Prisms: against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL
from paper_1504_01023_gb300 import api, build, meshgen
from test_fixed_algorithm import reference, rel
from test_fixed_even import _diffusion, _entry_errors, _points, _tets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = api.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("eps", [2.0 ** -9, 2.0 ** -20, 2.0 ** -30])
@pytest.mark.parametrize("four", [0, 1])
@pytest.mark.parametrize("route", ["aos", "soa", "nodes", "host"])
def test_tets(ctx, route, four, eps):
    nodes, conn = meshgen.tet_cube_indexed(12, 0.2, seed=1)
    x = nodes[conn]
    n = len(x)
    c = _diffusion(n, 1, (eps, 1.0, eps))[:, 0]
    even = np.arange(n) % 7 == 0
    c[even] = meshgen.generic_coefs(n, seed=2)[even]
    quad = api.QUAD_TET4 if four else api.QUAD_TET1
    kw = dict(kind=api.GENERIC, quad=quad, coef_mode=api.PER_ELEMENT, prec=api.FP64)
    X, C = torch.from_numpy(x), torch.from_numpy(c)
    if route == "soa":
        A = ctx.integrate(api.TET, X.reshape(n, -1).T.contiguous().cuda(), C.T.contiguous().cuda(), layout=api.SOA,
                          out_layout=api.SOA, **kw)[0].T.reshape(n, 4, 4)
    elif route == "nodes":
        A = ctx.integrate(api.TET, torch.from_numpy(nodes).cuda(), C.cuda(), layout=api.INDEXED, out_layout=api.AOS,
                          conn=torch.from_numpy(conn).cuda(), **kw)[0]
    elif route == "host":
        A = ctx.integrate(api.TET, X.pin_memory(), C.pin_memory(), layout=api.AOS, out_layout=api.AOS, **kw)[0]
    else:
        A = ctx.integrate(api.TET, X.cuda(), C.cuda(), layout=api.AOS, out_layout=api.AOS, **kw)[0]
    ctx.sync()
    A, ref, dbl = A.cpu().numpy(), reference(x, c, four, np.longdouble)[0], reference(x, c, four, np.float64)[0]
    for part in (even, ~even):
        assert np.quantile(_entry_errors(A[part], ref[part]), 0.99) <= 4 * np.quantile(_entry_errors(dbl[part], ref[part]), 0.99)


@pytest.mark.parametrize("eps", [2.0 ** -8, 2.0 ** -20])
@pytest.mark.parametrize("pq", [0, 1])
@pytest.mark.parametrize("route", ["pair", "soa"])
def test_prisms(ctx, route, pq, eps):
    x = meshgen.prism_slab_mesh(20, seed=1)
    n = len(x)
    c = _diffusion(n, 6 if pq else 1, (1.0, eps, eps))
    even = np.arange(n) % 7 == 0
    c[even] = meshgen.generic_coefs(n, 6 if pq else 1, seed=2).reshape(c.shape)[even]
    Ao, bo, _ = oracle.integrate(oracle.PRISM, api.GENERIC, oracle.Q_PRISM6, x, c if pq else c[:, 0], coef_per_q=bool(pq),
                                 n_threads=8)
    kw = dict(kind=api.GENERIC, quad=api.QUAD_PRISM6, coef_mode=api.PER_QPOINT if pq else api.PER_ELEMENT, prec=api.FP64)
    X, C = torch.from_numpy(x).cuda(), torch.from_numpy(c.reshape(n, -1)).cuda()
    if route == "soa":
        X, C = X.reshape(n, -1).T.contiguous(), C.T.contiguous()
        A, b, f = ctx.integrate(api.PRISM, X, C, layout=api.SOA, out_layout=api.SOA, **kw)
        A, b = A.T.reshape(n, 6, 6), b.T
    else:
        ctx.set_shape(32, 0, api.PRISM, X, C, layout=api.AOS, out_layout=api.AOS, tpe=2, **kw)
        A, b, f = ctx.integrate(api.PRISM, X, C, layout=api.AOS, out_layout=api.AOS, **kw)
    ctx.sync()
    assert oracle.rel_frobenius(A.cpu().numpy(), Ao).max() <= TOL[api.FP64]
    assert oracle.rel_frobenius(b.cpu().numpy(), bo).max() <= TOL[api.FP64]
    assert (f.cpu().numpy() == 0).all()


@pytest.mark.parametrize("kind", [api.POISSON, api.GENERIC])
@pytest.mark.parametrize("route", ["aos", "soa", "host"])
def test_stretched_tets(ctx, route, kind):
    """Tetrahedra stretched along directions of their own and ones with a long edge, mixed
    with ordinary ones: as near to the exact results as plain double evaluation, the
    median within a quarter, the 99% point within one bit (the kernels' double form sums in
    another order)."""
    n = 9000
    x = meshgen.tet_cube_mesh(12, seed=1)[:n].copy()
    odd = {name: np.arange(n) % 5 == i for i, name in ((1, "stretch"), (3, "long"))}
    for name, part in odd.items():
        x[part] = _tets(name, 5, n)[part]
    c = meshgen.generic_coefs(n, seed=2)
    C = torch.from_numpy(c if kind == api.GENERIC else c[:, 16:17].copy())
    X = torch.from_numpy(x)
    # (the four-point rule's summed weights are one unit in the last place off in b)
    kw = dict(kind=kind, quad=api.QUAD_TET4 if kind == api.GENERIC else api.QUAD_TET1, coef_mode=api.PER_ELEMENT,
              prec=api.FP64)
    if route == "soa":
        A, b, f = ctx.integrate(api.TET, X.reshape(n, -1).T.contiguous().cuda(), C.T.contiguous().cuda(), layout=api.SOA,
                                out_layout=api.SOA, **kw)
        A, b = A.T.reshape(n, 4, 4), b.T
    else:
        move = (lambda t: t.pin_memory()) if route == "host" else (lambda t: t.cuda())
        A, b, f = ctx.integrate(api.TET, move(X), move(C), layout=api.AOS, out_layout=api.AOS, **kw)
    ctx.sync()
    if kind == api.POISSON:
        c = np.zeros_like(c)
        c[:, [5, 10, 15]] = 1.0
        c[:, 16] = C.numpy()[:, 0]
    ref, dbl = reference(x, c, 1, np.longdouble), reference(x, c, 1, np.float64)
    for part in [np.arange(n) % 2 == 0] + list(odd.values()):
        for got, r, d in zip((A, b), ref, dbl):
            (mg, qg, _), (md, qd, _) = _points(rel(got.cpu().numpy(), r)[part]), _points(rel(d, r)[part])
            assert mg <= 1.25 * md and qg <= 2 * qd
    det = np.linalg.det(x[:, 1:] - x[:, :1])
    assert (f.cpu().numpy() == np.where(det < 0, 2, 0)).all()
