"""FP64 tetrahedra in pinned host memory, read and written in place over the host link
by the tile kernel (element-contiguous records on the device take the warp-at-a-time
kernel): the bits of the device call, at sizes around a tile of 32 elements and with
several tiles per block, records and results off their 16-byte boundaries, and elements
outside the fixed-point windows among ordinary ones; nothing around the results is
written."""
import numpy as np
import pytest
import torch

from paper_1504_01023_gb300 import api, build, meshgen

pytestmark = pytest.mark.gpu
CASES = [(api.GENERIC, api.QUAD_TET1, 0), (api.GENERIC, api.QUAD_TET4, 0), (api.POISSON, api.QUAD_TET1, 0),
         (api.POISSON, api.QUAD_TET1, 1), (api.POISSON, api.QUAD_TET4, 0), (api.POISSON, api.QUAD_TET4, 1)]


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _pinned(a, off):
    """A pinned copy of `a` that starts off * 8 bytes into its allocation, and that allocation."""
    t = torch.full((a.size + off + 4,), 77.0, dtype=torch.float64).pin_memory()
    v = t[off:off + a.size].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return t, v


def _check(ctx, kind, quad, cpq, n, in_off=0, out_off=0, shape=None):
    mesh = meshgen.tet_cube_mesh(12, seed=5)
    mesh = np.concatenate([mesh] * (n // len(mesh) + 1))[:n].copy()
    mesh[3::11] *= 2.0 ** 220                              # outside the windows
    mesh[5::13] = 1e-2 * np.arange(4.0)[:, None] + 1e-5 * mesh[5::13]
    mesh[7::17, 1] = mesh[7::17, 0]                        # degenerate
    nq = api.NQ[quad] if cpq else 1
    c = (meshgen.generic_coefs(n, 1, seed=6) if kind == api.GENERIC else
         meshgen.poisson_coefs(n, nq, value=None, seed=7)).reshape(n, -1).copy()
    kw = dict(kind=kind, quad=quad, coef_mode=api.PER_QPOINT if cpq else api.PER_ELEMENT, prec=api.FP64, layout=api.AOS,
              out_layout=api.AOS)
    ref = ctx.integrate(api.TET, torch.from_numpy(mesh).cuda(), torch.from_numpy(c).cuda(), **kw)
    ctx.sync()
    (_, X), (_, C) = _pinned(mesh, in_off), _pinned(c, in_off)
    (ka, A), (kb, b) = _pinned(np.zeros((n, 4, 4)), out_off), _pinned(np.zeros((n, 4)), out_off)
    flags = torch.full((n + 8,), 99, dtype=torch.uint8).pin_memory()
    out = (A, b, flags[:n])
    if shape:
        ctx.set_shape(shape[0], shape[1], api.TET, X, C, out=out, **kw)
    ctx.integrate(api.TET, X, C, out=out, **kw)
    for got, want in zip(out, ref):
        assert torch.equal(got, want.cpu())
    assert (flags[n:] == 99).all() and (flags[7:n:17] == 4).all()
    for t, v in ((ka, A), (kb, b)):
        assert (t[:out_off] == 77).all() and (t[out_off + v.numel():] == 77).all()


@pytest.mark.parametrize("kind,quad,cpq", CASES)
@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 1001])
def test_sizes(ctx, kind, quad, cpq, n):
    _check(ctx, kind, quad, cpq, n)


@pytest.mark.parametrize("kind,quad,cpq", CASES)
@pytest.mark.parametrize("in_off,out_off", [(1, 0), (0, 1), (1, 3)])
def test_alignment(ctx, kind, quad, cpq, in_off, out_off):
    _check(ctx, kind, quad, cpq, 1003, in_off, out_off)


@pytest.mark.parametrize("kind,quad,cpq", CASES)
def test_several_tiles_per_block(ctx, kind, quad, cpq):
    _check(ctx, kind, quad, cpq, 300007)


@pytest.mark.parametrize("kind,quad,cpq", CASES)
@pytest.mark.parametrize("shape", [(64, 0), (256, 1)])
def test_pinned_shapes(ctx, kind, quad, cpq, shape):
    with api.Context(0) as own:
        _check(own, kind, quad, cpq, 2003, shape=shape)
