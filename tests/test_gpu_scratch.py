"""The scratch of mixed and double-word calls (list and counter of the elements for the
double Jacobian pass) on the stream of the call, against the oracle: first calls of a
context and of its serving slots beside a default stream that is still busy; calls and
replays that overlap on several streams, and the calls that follow them alone."""
import time

import numpy as np
import pytest
import torch

from helpers import TOL, make_inputs, max_errors, run_oracle, to_device_inputs
from paper_1504_01023_gb300 import api, build, meshgen

pytestmark = pytest.mark.gpu
KW = dict(kind=api.GENERIC, quad=api.QUAD_TET4, coef_mode=api.PER_ELEMENT, layout=api.AOS, out_layout=api.AOS)
BUSY = 1 << 29     # clocks of a waiting kernel: about a quarter of a second


class Case:
    """n tetrahedra, a tenth of them slivers, with outputs and the oracle's results."""

    def __init__(self, n, prec, seed):
        mesh = meshgen.tet_cube_mesh(16, seed=seed)[:n].copy()
        self.flagged = meshgen.make_slivers(mesh, 0.1, seed=seed + 1)
        mesh, c = make_inputs(api.TET, api.GENERIC, api.QUAD_TET4, 0, seed=seed, mesh=mesh)
        self.n, self.prec = n, prec
        self.X, self.C, c_used = to_device_inputs(api.TET, mesh, c, prec, api.AOS)
        self.out = api.alloc_out(api.TET, n, prec, api.AOS, self.X.device)
        self.ref = run_oracle(api.TET, api.GENERIC, api.QUAD_TET4, 0, mesh, c_used)[:2]

    def call(self, ctx, stream=None):
        ctx.integrate(api.TET, self.X, self.C, prec=self.prec, out=self.out, stream=stream, **KW)

    def check(self, out=None):
        A, b, f = (t.cpu().numpy() for t in (out or self.out))
        ea, eb = max_errors(A.astype(np.float64), b.astype(np.float64), *self.ref)
        assert ea <= TOL[self.prec] and eb <= TOL[self.prec]
        assert (f[self.flagged] & 1).mean() > 0.5


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()
    with api.Context(0) as ctx:            # modules loaded before the timed kernels below
        for prec in (api.FP32_MIXED, api.FP64_DW):
            Case(100, prec, 3).call(ctx)
        ctx.sync()


@pytest.mark.parametrize("prec", [api.FP32_MIXED, api.FP64_DW])
def test_first_call_beside_a_busy_default_stream(prec):
    first, second = Case(20001, prec, 11), Case(7003, prec, 21)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(BUSY)
    with api.Context(0) as ctx:
        first.call(ctx, side)
        second.call(ctx, side)
        side.synchronize()
        first.check()
        second.check()
        ctx.sync()


def test_first_served_requests_beside_a_busy_default_stream():
    case = Case(20001, api.FP64_DW, 12)
    with api.Context(0) as ctx:
        mid = ctx.mesh_register(api.TET, case.X, api.AOS)
        torch.cuda.synchronize()
        torch.cuda._sleep(BUSY)
        tickets = [ctx.serve_submit(mid, api.GENERIC, api.QUAD_TET4, api.PER_ELEMENT, case.C, prec=api.FP64_DW)
                   for _ in range(8)]
        deadline = time.time() + 60
        for t in tickets:
            r = ctx.serve_poll(t)
            while r is None and time.time() < deadline:
                time.sleep(1e-3)
                r = ctx.serve_poll(t)
            assert r is not None and r.status == 0
            case.check(ctx.serve_result_tensors(t, r))
            ctx.serve_release(t)
        ctx.mesh_release(mid)
        ctx.sync()


def _alone(ctx, cases):
    """Calls with nothing else on the device, and a matrix-free product (which adds an
    element twice if its fix-up list holds entries of an earlier call)."""
    for case in cases:
        for t in case.out:
            t.zero_()
        case.call(ctx)
        ctx.sync()
        case.check()
        n, (Ao, bo) = case.n, case.ref
        nodes = case.X.reshape(-1, 3)
        conn = torch.arange(4 * n, dtype=torch.int32, device="cuda").reshape(n, 4)
        dt = torch.float32 if case.prec == api.FP32_MIXED else torch.float64
        y, f = torch.zeros(4 * n, dtype=dt, device="cuda"), torch.zeros(4 * n, dtype=dt, device="cuda")
        ctx.apply(api.TET, nodes, conn, case.C, api.GENERIC, api.QUAD_TET4, torch.ones_like(y), y, f, prec=case.prec)
        ctx.sync()
        # row sums of A: four entries, each within the form's tolerance of the element's norm
        ey = np.abs(y.cpu().numpy().reshape(n, 4) - Ao.sum(2)).max(1) / np.linalg.norm(Ao, axis=(1, 2))
        assert ey.max() <= 4 * TOL[case.prec]
        assert max_errors(Ao, f.cpu().numpy().reshape(n, 4).astype(np.float64), Ao, bo)[1] <= TOL[case.prec]


@pytest.mark.parametrize("prec", [api.FP32_MIXED, api.FP64_DW])
def test_calls_overlapping_on_two_streams(prec):
    cases = [Case(20001, prec, 31), Case(1003, prec, 32)]
    streams = [torch.cuda.Stream() for _ in cases]
    torch.cuda.synchronize()
    with api.Context(0) as ctx:
        for _ in range(100):
            for case, s in zip(cases, streams):
                case.call(ctx, s)
        torch.cuda.synchronize()
        for case in cases:
            case.check()
        _alone(ctx, cases)


@pytest.mark.parametrize("prec", [api.FP32_MIXED, api.FP64_DW])
def test_replays_overlapping_plain_calls(prec):
    captured, plain = Case(20001, prec, 41), Case(1003, prec, 42)
    larger = Case(24000, prec, 43)       # its capture outgrows the first graph's list
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with api.Context(0) as ctx:
        graphs = []
        for case in (captured, larger):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                case.call(ctx, s)
                case.call(ctx, s)
            graphs.append(g)
        for _ in range(50):
            with torch.cuda.stream(s):
                for g in graphs:
                    g.replay()
            plain.call(ctx, t)
            plain.call(ctx, t)
        torch.cuda.synchronize()
        for case in (captured, larger, plain):
            case.check()
        _alone(ctx, [plain, captured])


def test_more_streams_than_scratch():
    cases = [Case(500 + 211 * i, api.FP32_MIXED, 50 + i) for i in range(24)]
    streams = [torch.cuda.Stream() if i % 3 else torch.cuda.Stream(priority=-1) for i in range(24)]
    torch.cuda.synchronize()
    with api.Context(0) as ctx:
        for order in (range(24), reversed(range(24)), range(0, 24, 2)):
            for i in order:
                cases[i].call(ctx, streams[i])
        torch.cuda.synchronize()
        for case in cases:
            case.check()
        _alone(ctx, cases[:2])
