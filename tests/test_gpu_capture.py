"""Calls captured in a CUDA graph and replayed: each replay is a whole call (its
fix-up list starts empty whatever ran before it), on the inputs of that moment, and
calls between replays do not disturb it."""
import numpy as np
import pytest
import torch

from helpers import TOL, make_inputs, max_errors, run_oracle, to_device_inputs
from paper_1504_01023_gb300 import api, build, meshgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [api.FP64, api.FP32_MIXED, api.FP64_DW])
@pytest.mark.parametrize("layout", [api.AOS, api.SOA])
def test_replays_are_whole_calls(prec, layout):
    build.build()
    n = 3001
    mesh = meshgen.tet_cube_mesh(8, seed=3)[:n]
    flagged = meshgen.make_slivers(mesh, 0.1, seed=4)
    mesh, c = make_inputs(api.TET, api.GENERIC, api.QUAD_TET4, 0, seed=3, mesh=mesh)
    X, C, c_used = to_device_inputs(api.TET, mesh, c, prec, layout)
    X2 = X.clone()
    out = api.alloc_out(api.TET, n, prec, layout, X.device)
    kw = dict(kind=api.GENERIC, quad=api.QUAD_TET4, coef_mode=api.PER_ELEMENT, prec=prec, layout=layout,
              out_layout=layout, out=out)
    ref = [run_oracle(api.TET, api.GENERIC, api.QUAD_TET4, 0, m, c_used)[:2] for m in (mesh, 0.5 * mesh)]

    def check(i):
        A, b, f = (t.cpu().numpy() for t in out)
        if layout == api.SOA:
            A, b = A.T.reshape(n, 4, 4), b.T
        ea, eb = max_errors(A.astype(np.float64), b.astype(np.float64), *ref[i])
        assert ea <= TOL[prec] and eb <= TOL[prec]
        if prec != api.FP64:
            assert (f[flagged] & 1).mean() > 0.5 and (f & 1).sum() < 0.2 * n

    with api.Context(0) as ctx:
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            ctx.integrate(api.TET, X, C, **kw)          # scratch in place
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ctx.integrate(api.TET, X, C, **kw)
            ctx.integrate(api.TET, X, C, **kw)
        for i, src in enumerate((X2, 0.5 * X2, X2)):
            X.copy_(src)
            for t in out:
                t.zero_()
            g.replay()
            torch.cuda.synchronize()
            check(i % 2)
            ctx.integrate(api.TET, X, C, **kw)
            ctx.sync()
            check(i % 2)
