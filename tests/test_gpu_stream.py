"""The warp-at-a-time kernel of FP64 tetrahedra (element-contiguous records): sizes
around a warp's 32 elements and a block's tile, persistent blocks that run over
several tiles, records and results off their 16- and 32-byte boundaries, and warps
that mix ordinary elements with elements outside the fixed-point windows, against
the oracle (1e-12 per element, the FP64 form's tolerance); nothing outside the
result arrays is written."""
import numpy as np
import pytest
import torch

import oracle
from helpers import ORACLE_RULE, TOL
from paper_1504_01023_gb300 import api, build, meshgen

pytestmark = pytest.mark.gpu
CASES = [(api.GENERIC, api.QUAD_TET4, 0), (api.GENERIC, api.QUAD_TET1, 0), (api.POISSON, api.QUAD_TET1, 0),
         (api.POISSON, api.QUAD_TET4, 1)]


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _inputs(n, kind, quad, cpq, odd):
    mesh = meshgen.tet_cube_mesh(12, seed=5)[:n].copy()
    nq = api.NQ[quad] if cpq else 1
    c = (meshgen.generic_coefs(n, 1, seed=6) if kind == api.GENERIC else
         meshgen.poisson_coefs(n, nq, value=None, seed=7)).reshape(n, -1).copy()
    if odd:      # outside the windows: scaled far away, a needle, degenerate
        mesh[3::11] *= 2.0 ** 220      # (the double form squares cofactors: they stay below 2^512)
        s = mesh[5::13]
        s[:] = 1e-2 * np.arange(4.0)[:, None] + 1e-5 * s     # along (1, 1, 1)
        mesh[7::17, 1] = mesh[7::17, 0]
    return mesh, c


def _shifted(a, off):
    """A device copy of `a` that starts off * 8 bytes into its allocation."""
    t = torch.full((a.size + off + 4,), 77.0, dtype=torch.float64, device="cuda")
    v = t[off:off + a.size].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return t, v


@pytest.mark.parametrize("kind,quad,cpq", CASES)
@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 65, 127, 513, 4099])
@pytest.mark.parametrize("shape", [(32, 0), (64, 1), (512, 1)])
def test_sizes_and_shapes(ctx, kind, quad, cpq, n, shape):
    _check(ctx, kind, quad, cpq, n, shape, 0, 0, False)


@pytest.mark.parametrize("kind,quad,cpq", CASES)
@pytest.mark.parametrize("in_off,out_off", [(1, 0), (0, 1), (0, 2), (1, 3)])
def test_alignment(ctx, kind, quad, cpq, in_off, out_off):
    _check(ctx, kind, quad, cpq, 1001, (128, 1), in_off, out_off, False)


@pytest.mark.parametrize("kind,quad,cpq", CASES)
@pytest.mark.parametrize("in_off", [0, 1])
def test_elements_outside_the_windows(ctx, kind, quad, cpq, in_off):
    _check(ctx, kind, quad, cpq, 2003, (64, 1), in_off, 0, True)


def test_many_tiles_per_block(ctx):
    _check(ctx, api.GENERIC, api.QUAD_TET4, 0, 10301, (32, 1), 0, 0, True, reps=60)


def _max_error(v, ref):
    """oracle.rel_frobenius, each element scaled first (entries up to 2^640 here)."""
    s = np.abs(ref).reshape(len(ref), -1).max(1)
    s = np.where(s > 0, s, 1.0).reshape((-1,) + (1,) * (ref.ndim - 1))
    return oracle.rel_frobenius(v / s, ref / s).max()


def _check(ctx, kind, quad, cpq, n, shape, in_off, out_off, odd, reps=1):
    mesh, c = _inputs(n, kind, quad, cpq, odd)
    Ao, bo, _ = oracle.integrate(oracle.TET, kind, ORACLE_RULE[quad], mesh, c, coef_per_q=bool(cpq), n_threads=8)
    if reps > 1:   # more tiles than resident blocks
        mesh, c, Ao, bo = (np.concatenate([v] * reps) for v in (mesh, c, Ao, bo))
        n *= reps
    kx, X = _shifted(mesh, in_off)
    kc, C = _shifted(c, in_off)
    ka, A = _shifted(np.zeros((n, 4, 4)), out_off)
    kb, b = _shifted(np.zeros((n, 4)), out_off)
    flags = torch.full((n + 8,), 99, dtype=torch.uint8, device="cuda")
    kw = dict(kind=kind, quad=quad, coef_mode=api.PER_QPOINT if cpq else api.PER_ELEMENT, prec=api.FP64,
              layout=api.AOS, out_layout=api.AOS, out=(A, b, flags[:n]))
    ctx.set_shape(shape[0], shape[1], api.TET, X, C, **kw)
    ctx.integrate(api.TET, X, C, **kw)
    ctx.sync()
    keep = np.ones(n, dtype=bool)
    if odd:
        keep[np.arange(n) % (n // reps) % 13 == 5] = False
    assert _max_error(A.cpu().numpy()[keep], Ao[keep]) <= TOL[api.FP64]
    assert _max_error(b.cpu().numpy()[keep], bo[keep]) <= TOL[api.FP64]
    det = np.linalg.det(mesh[:, 1:] - mesh[:, :1])
    if odd:
        # every element, the needles (too ill-conditioned for the oracle's tolerance)
        # included: the same bits as through the tile kernel
        As, bs, fs = ctx.integrate(api.TET, X.reshape(n, -1).T.contiguous(), C.T.contiguous(), kind, quad,
                                   kw["coef_mode"], api.FP64, api.SOA, api.SOA)
        ctx.sync()
        assert torch.equal(As.T.reshape(n, 4, 4), A) and torch.equal(bs.T, b) and torch.equal(fs, flags[:n])
    else:
        assert (flags[:n].cpu().numpy() == np.where(det < 0, 2, 0)).all()
    assert (flags[n:] == 99).all()
    for t, v in ((ka, A), (kb, b)):
        assert (t[:out_off] == 77).all() and (t[out_off + v.numel():] == 77).all()
