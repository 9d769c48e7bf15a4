"""Tuning-cache files: a line of an earlier build, which names no revision, keeps its
shape where the kernels are the same or no tuner is on; for the FP64 form, whose kernels
changed since, a tuner chooses again and saves the line with a revision."""
import pytest

from helpers import TOL, make_inputs, max_errors, run_oracle, to_device_inputs
from paper_1504_01023_gb300 import api, build

pytestmark = pytest.mark.gpu
FORMS = (api.FP64, api.FP32_MIXED)


def _lines(path):
    with open(path) as f:
        return {t[1]: t for t in (line.split() for line in f)}


def test_lines_of_an_earlier_build(tmp_path):
    build.build()
    path = str(tmp_path / "shapes")
    n = 3000
    mesh, c = make_inputs(api.PRISM, api.POISSON, api.QUAD_PRISM6, 1, n=n, seed=5)
    kw = {p: dict(kind=api.POISSON, quad=api.QUAD_PRISM6, coef_mode=api.PER_QPOINT, prec=p, layout=api.AOS,
                  out_layout=api.AOS) for p in FORMS}
    data = {p: to_device_inputs(api.PRISM, mesh, c, p, api.AOS) for p in FORMS}

    def run(ctx, p):
        X, C, used = data[p]
        A, b, f = ctx.integrate(api.PRISM, X, C, **kw[p])
        ctx.sync()
        ea, eb = max_errors(A.double().cpu().numpy(), b.double().cpu().numpy(),
                            *run_oracle(api.PRISM, api.POISSON, api.QUAD_PRISM6, 1, mesh, used)[:2])
        assert ea <= TOL[p] and eb <= TOL[p]
        return ctx.shape(api.PRISM, X, C, **kw[p])

    with api.Context(0, autotune=True, tuning_cache=path) as ctx:
        tuned = {p: run(ctx, p) for p in FORMS}
    saved = _lines(path)
    assert len(saved) == 2 and all(len(t) == 6 and t[5] == "2" for t in saved.values())
    key = {p: next(k for k in saved if f"p{p}q" in k) for p in FORMS}
    # the same file as an earlier build left it, with a shape that is not the tuned one
    old = {p: next(s for s in ((64, 0, 1), (32, 1, 1)) if s != tuned[p]) for p in FORMS}
    device = saved[key[FORMS[0]]][0]
    with open(path, "w") as f:
        for p in FORMS:
            f.write(" ".join([device, key[p]] + [str(v) for v in old[p]]) + "\n")
    with api.Context(0, autotune=False, tuning_cache=path) as ctx:
        assert all(run(ctx, p) == old[p] for p in FORMS)
        X, C, _ = data[api.FP64]
        ctx.set_shape(32, 0, api.PRISM, X[:100], C[:100], **kw[api.FP64])     # writes the file
    assert _lines(path)[key[api.FP64]][2:] == [str(v) for v in old[api.FP64]] + ["1"]
    with api.Context(0, autotune=True, tuning_cache=path) as ctx:
        assert run(ctx, api.FP32_MIXED) == old[api.FP32_MIXED]
        run(ctx, api.FP64)
    again = _lines(path)
    assert again[key[api.FP64]][5] == "2" and again[key[api.FP32_MIXED]][5] == "1"
