"""Workloads of the integration library, as programs that use it run them.

``listed()`` names twelve of them, ``draw(rng)`` gives more of the same ranges.
``prepare`` makes what a program holds before the call (meshes, coefficients,
output buffers, the context), ``run`` makes one call, ``exact`` gives the same
outputs by plain float64 quadrature in torch.

Meshes are jittered Kuhn cubes (tetrahedra) and jittered extruded slabs
(prisms), numbered cube by cube; coefficients are independent draws per element
or per integration point: diffusion Q diag(l) Q^T with l in [0.1, 10],
convection and sources in [-1, 1], reaction in [0, 1].
"""
from __future__ import annotations

import math

import torch

from paper_1504_01023_gb300 import api

_ET = {"tet": api.TET, "prism": api.PRISM}
_KIND = {"poisson": api.POISSON, "generic": api.GENERIC}
_PREC = {"fp64": api.FP64, "mixed": api.FP32_MIXED, "dw": api.FP64_DW}
_QUAD = {"tet1": api.QUAD_TET1, "tet4": api.QUAD_TET4, "prism6": api.QUAD_PRISM6}
_MODE = {"element": api.PER_ELEMENT, "point": api.PER_QPOINT}
_LAYOUT = {"aos": api.AOS, "soa": api.SOA}


def _case(name, call, et, kind, quad, mode, prec, n, layout="aos", slivers=0.0):
    c = {"call": call, "et": et, "kind": kind, "quad": quad, "mode": mode, "prec": prec, "n": n, "layout": layout,
         "slivers": slivers}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest mesh of the batched mix on its own: one call's latency
        _case("tet_generic_mixed_1k", "integrate", "tet", "generic", "tet4", "element", "mixed", 1000),
        # Laplace operator on 20^3 cubes as the paper's Poisson problem is stated: a few microseconds of work
        _case("tet_poisson_fp64_48k", "integrate", "tet", "poisson", "tet1", "element", "fp64", 48000),
        # the same problem on a mesh that fills the GPU
        _case("tet_poisson_fp64_2m", "integrate", "tet", "poisson", "tet1", "element", "fp64", 2000000),
        # convection-diffusion-reaction on 100^3 cubes in double, the headline workload (largest)
        _case("tet_generic_fp64_6m", "integrate", "tet", "generic", "tet4", "element", "fp64", 6000000),
        # the same in the mixed form, bound by memory
        _case("tet_generic_mixed_6m", "integrate", "tet", "generic", "tet4", "element", "mixed", 6000000),
        # plane-major arrays (the default layout) of an odd length, a mesh with 1% slivers for the double Jacobian pass
        _case("tet_generic_mixed_soa_slivers", "integrate", "tet", "generic", "tet4", "element", "mixed", 399999, "soa",
              0.01),
        # double accuracy on the float pipes, a ragged size
        _case("tet_generic_dw_1m", "integrate", "tet", "generic", "tet4", "element", "dw", 1000003),
        # one product of a Krylov solver with the operator that is never assembled, on a node table
        _case("tet_generic_apply_3m", "apply", "tet", "generic", "tet4", "element", "mixed", 3000000),
        # Laplace operator on prisms in double, the load varying over the element
        _case("prism_poisson_fp64_500k", "integrate", "prism", "poisson", "prism6", "point", "fp64", 500000),
        # convection-diffusion-reaction on prisms in double, coefficients per integration point, a ragged size
        _case("prism_generic_fp64_300k", "integrate", "prism", "generic", "prism6", "point", "fp64", 300001),
        # the 1000 x 1000 slab of generic prisms in the mixed form
        _case("prism_generic_mixed_2m", "integrate", "prism", "generic", "prism6", "point", "mixed", 2000000),
        # many small and middling meshes of all kinds in one submission, replayed as a time-stepping program does
        {"name": "batch_mixed_64", "call": "batch", "meshes": 64, "lo": 1000, "hi": 500000, "pick": 4},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["tet", "tet", "tet", "prism", "prism", "apply", "nodes", "batch"])
    if what == "batch":
        return {"call": "batch", "meshes": rng.randint(8, 64), "lo": 1000, "hi": size(50000, 500000),
                "pick": rng.randint(0, 1 << 20)}
    prec = rng.choice(["fp64", "fp64", "mixed", "dw"])
    kind = rng.choice(["poisson", "generic"])
    if what in ("apply", "nodes"):
        return _case(None, what, "tet", kind, rng.choice(["tet1", "tet4"]), "element", prec, size(1000, 2000000))
    layout = rng.choice(["aos", "aos", "soa"])
    if what == "tet":
        slivers = rng.choice([0.0, 0.0, 0.01]) if prec == "mixed" else 0.0
        return _case(None, "integrate", "tet", kind, rng.choice(["tet1", "tet4"]), "element", prec,
                     size(1000, 4000000), layout, slivers)
    hi = 2000000 if prec == "mixed" else 300000
    return _case(None, "integrate", "prism", kind, "prism6", rng.choice(["element", "point"]), prec, size(1000, hi),
                 layout)


# ---------------------------------------------------------------------------
# Inputs, on the GPU, from the seed alone
# ---------------------------------------------------------------------------
_DEV = "cuda"
# Kuhn split of a cube into six positively oriented tetrahedra around its main diagonal
_PERMS = [((0, 1, 2), 0), ((1, 2, 0), 0), ((2, 0, 1), 0), ((0, 2, 1), 1), ((2, 1, 0), 1), ((1, 0, 2), 1)]


def _corners():
    out = []
    for perm, odd in _PERMS:
        v = [[0, 0, 0]]
        for ax in perm:
            w = list(v[-1])
            w[ax] += 1
            v.append(w)
        if odd:
            v[1], v[2] = v[2], v[1]
        out.append(v)
    return torch.tensor(out, device=_DEV)


def _rand(gen, lo, hi, *shape):
    return torch.rand(shape, generator=gen, device=_DEV, dtype=torch.float64) * (hi - lo) + lo


def _tet_mesh(n, gen):
    """(nodes [N, 3], conn [n, 4]): the first n tetrahedra of the smallest cube that holds them."""
    k = 1
    while 6 * k ** 3 < n:
        k += 1
    m, h = k + 1, 1.0 / k
    i = torch.arange(m, device=_DEV)
    z, y, x = torch.meshgrid(i, i, i, indexing="ij")
    nodes = torch.stack([x, y, z], -1).reshape(-1, 3).double() * h
    nodes += _rand(gen, -0.2 * h, 0.2 * h, *nodes.shape)
    cube = torch.arange((n + 5) // 6, device=_DEV)
    base = cube % k + m * ((cube // k) % k + m * (cube // (k * k)))
    off = _corners()
    off = off[..., 0] + m * (off[..., 1] + m * off[..., 2])
    conn = (base[:, None, None] + off[None]).reshape(-1, 4)[:n]
    return nodes, conn.int().contiguous()


def _prism_mesh(n, gen):
    """(nodes, conn [n, 6]): the first n prisms of the smallest square slab that holds them."""
    k = 1
    while 2 * k * k < n:
        k += 1
    m, h = k + 1, 1.0 / k
    i = torch.arange(m, device=_DEV)
    y, x = torch.meshgrid(i, i, indexing="ij")
    xy = torch.stack([x, y], -1).reshape(-1, 2).double() * h
    zb = _rand(gen, -0.1 * h, 0.1 * h, m * m, 1)
    zt = h + _rand(gen, -0.1 * h, 0.1 * h, m * m, 1)
    nodes = torch.cat([torch.cat([xy, zb], 1), torch.cat([xy, zt], 1)])
    sq = torch.arange((n + 1) // 2, device=_DEV)
    p = sq % k + m * (sq // k)
    tri = torch.stack([torch.stack([p, p + 1, p + 1 + m], -1), torch.stack([p, p + 1 + m, p + m], -1)], 1)
    tri = tri.reshape(-1, 3)[:n]
    return nodes, torch.cat([tri, tri + m * m], 1).int().contiguous()


def _flatten(x, fraction, gen):
    """Slivers: vertex 3 of a random subset moved to t times its height, t log-uniform in [2e-3, 2e-2]."""
    k = int(round(fraction * x.shape[0]))
    idx = torch.randperm(x.shape[0], generator=gen, device=_DEV)[:k]
    t = torch.exp(_rand(gen, math.log(2e-3), math.log(2e-2), k, 1))
    c = x[idx, :3].mean(1)
    x[idx, 3] = c + t * (x[idx, 3] - c)


def _coefs(case, gen):
    """[n, points, 1 or 20], float64."""
    n = case["n"]
    nq = {"tet1": 1, "tet4": 4, "prism6": 6}[case["quad"]] if case["mode"] == "point" else 1
    if case["kind"] == "poisson":
        if nq == 1:
            return torch.ones(n, 1, 1, device=_DEV, dtype=torch.float64)
        return _rand(gen, -1, 1, n, nq, 1)
    q = torch.randn(n, nq, 4, generator=gen, device=_DEV, dtype=torch.float64)
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    rot = [[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
           [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
           [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]]
    lam = _rand(gen, 0.1, 10, n, nq, 3)
    c = _rand(gen, -1, 1, n, nq, 20)
    c[..., 0].abs_()
    for i in range(3):
        for j in range(3):
            c[..., 4 * i + j + 5] = sum(rot[i][k] * lam[..., k] * rot[j][k] for k in range(3))
    return c


def _inputs(case, seed):
    """(nodes, conn, element coordinates [n, NS, 3], coefficients [n, points, k] as the program holds them)."""
    gen = torch.Generator(_DEV)
    gen.manual_seed(seed)
    nodes, conn = (_tet_mesh if case["et"] == "tet" else _prism_mesh)(case["n"], gen)
    x = nodes[conn.long()]
    if case["slivers"]:
        _flatten(x, case["slivers"], gen)
    c = _coefs(case, gen)
    return nodes, conn, x, c.float() if case["prec"] == "mixed" else c, gen


def _meshes(case):
    """The meshes of a batched case: sizes log-uniform, types and kinds half and half."""
    g = torch.Generator()
    g.manual_seed(case["pick"])
    out = []
    for _ in range(case["meshes"]):
        u, t, k = torch.rand(3, generator=g).tolist()
        n = int(round(math.exp(math.log(case["lo"]) + u * math.log(case["hi"] / case["lo"]))))
        kind = "poisson" if k < 0.5 else "generic"
        if t < 0.5:
            out.append(_case(None, "integrate", "tet", kind, "tet1" if k < 0.5 else "tet4", "element", "mixed", n))
        else:
            out.append(_case(None, "integrate", "prism", kind, "prism6", "point", "mixed", n))
    return out


def _offsets(meshes):
    """Each mesh's (first, end) in the program's arrays of A, b and flags, its parts on 16-byte boundaries, and the
    arrays' lengths."""
    at, offs = [0, 0, 0], []
    for c in meshes:
        ns = api.NS[_ET[c["et"]]]
        offs.append([(a, a + c["n"] * k) for a, k in zip(at, (ns * ns, ns, 1))])
        at = [-(-end // 16) * 16 for _, end in offs[-1]]
    return offs, at


_context = None


def _ctx():
    """The program's one context; launch shapes are tuned on the first call of a size class and kept."""
    global _context
    if _context is None:
        _context = api.Context(torch.cuda.current_device(), autotune=True)
    return _context


def _enums(case):
    return _ET[case["et"]], _KIND[case["kind"]], _QUAD[case["quad"]], _MODE[case["mode"]], _PREC[case["prec"]]


def prepare(case, seed):
    ctx = _ctx()
    if case["call"] == "batch":
        meshes = _meshes(case)
        offs, total = _offsets(meshes)
        out = [torch.zeros(k, device=_DEV, dtype=t) for k, t in zip(total, (torch.float32, torch.float32, torch.uint8))]
        items, keep = [], []
        for i, (c, o) in enumerate(zip(meshes, offs)):
            et, kind, quad, mode, prec = _enums(c)
            _, _, x, cf, _ = _inputs(c, seed * 1000 + i)
            cf = cf.reshape(c["n"], -1)
            items.append((et, api.make_args(et, x, cf, kind, quad, mode, prec, api.AOS),
                          api.make_out(*(t[a:b] for t, (a, b) in zip(out, o)), api.AOS)))
            keep.append((x, cf))
        return {"case": case, "ctx": ctx, "items": items, "keep": keep, "out": out}
    et, kind, quad, mode, prec = _enums(case)
    nodes, conn, x, c, gen = _inputs(case, seed)
    c = c.reshape(case["n"], -1)
    st = {"case": case, "ctx": ctx, "c": c}
    if case["call"] == "apply":
        st.update(nodes=nodes, conn=conn, x=_rand(gen, -1, 1, nodes.shape[0]).to(c.dtype))
        st["y"] = torch.empty_like(st["x"])
        st["f"] = torch.empty_like(st["x"])
        return st
    if case["call"] == "nodes":
        st.update(nodes=nodes, conn=conn, out=api.alloc_out(et, case["n"], prec, api.AOS, x.device))
        return st
    lay = _LAYOUT[case["layout"]]
    if lay == api.SOA:
        x = x.reshape(case["n"], -1).T.contiguous()
        st["c"] = c.T.contiguous()
    st.update(x=x, out=api.alloc_out(et, case["n"], prec, lay, x.device))
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["call"] == "batch":
        ctx.batch_submit(state["items"])
        return state["out"]
    et, kind, quad, mode, prec = _enums(case)
    if case["call"] == "apply":
        y, f = state["y"].zero_(), state["f"].zero_()
        ctx.apply(et, state["nodes"], state["conn"], state["c"], kind, quad, state["x"], y, f, mode, prec)
        return y, f
    if case["call"] == "nodes":
        return ctx.integrate(et, state["nodes"], state["c"], kind, quad, mode, prec, api.INDEXED, api.AOS,
                             out=state["out"], conn=state["conn"])
    lay = _LAYOUT[case["layout"]]
    return ctx.integrate(et, state["x"], state["c"], kind, quad, mode, prec, lay, lay, out=state["out"])


def work(case):
    if case["call"] == "batch":
        per = [work(c) for c in _meshes(case)]
        return {k: sum(p[k] for p in per) for k in ("bytes", "flops")}
    et, kind, quad, mode, prec = _enums(case)
    n, ns, scalar = case["n"], api.NS[et], 4 if prec == api.FP32_MIXED else 8
    # one multiply-add counts two: Jacobian terms, coefficient products and accumulation with loop-invariant terms
    # taken out, per element
    flops = {("tet", "poisson"): 110, ("tet", "generic"): 310, ("prism", "poisson"): 900,
             ("prism", "generic"): 2900}[(case["et"], case["kind"])]
    coefs = api.n_coefs(kind, quad, mode) * scalar
    if case["call"] in ("apply", "nodes"):
        k = 1
        while 6 * k ** 3 < n:
            k += 1
        nodes = (k + 1) ** 3
        if case["call"] == "apply":
            return {"bytes": n * (4 * ns + coefs) + nodes * (24 + 3 * scalar), "flops": n * (flops + 2 * ns * ns)}
        return {"bytes": n * (4 * ns + coefs + (ns * ns + ns) * scalar + 1) + nodes * 24, "flops": n * flops}
    return {"bytes": n * (24 * ns + coefs + (ns * ns + ns) * scalar + 1), "flops": n * flops}


# ---------------------------------------------------------------------------
# The same outputs by the plain quadrature sum in float64
# ---------------------------------------------------------------------------
def _rule(quad):
    """(weights, shape values [q][r], reference derivatives [q][r][3])"""
    if quad in ("tet1", "tet4"):
        a, b = (5 - math.sqrt(5)) / 20, (5 + 3 * math.sqrt(5)) / 20
        pts = [[0.25] * 4] if quad == "tet1" else [[b if r == q else a for r in range(4)] for q in range(4)]
        d = [[-1, -1, -1], [1, 0, 0], [0, 1, 0], [0, 0, 1]]
        return [1 / 6 / len(pts)] * len(pts), pts, [d] * len(pts)
    w, phi, der = [], [], []
    for z in (-1 / math.sqrt(3), 1 / math.sqrt(3)):
        for t in range(3):
            lam = [2 / 3 if k == t else 1 / 6 for k in range(3)]
            dl = [[-1, -1], [1, 0], [0, 1]]
            zb, zt = (1 - z) / 2, (1 + z) / 2
            w.append(1 / 6)
            phi.append([v * zb for v in lam] + [v * zt for v in lam])
            der.append([[d[0] * zb, d[1] * zb, -v / 2] for d, v in zip(dl, lam)] +
                       [[d[0] * zt, d[1] * zt, v / 2] for d, v in zip(dl, lam)])
    return w, phi, der


def _integrate_exact(case, x, c):
    """A [n, NS, NS], b [n, NS] from coordinates [n, NS, 3] and coefficients [n, points, k]."""
    n, ns = x.shape[:2]
    A = torch.zeros(n, ns, ns, device=x.device, dtype=torch.float64)
    b = torch.zeros(n, ns, device=x.device, dtype=torch.float64)
    rule = _rule(case["quad"])
    for s in range(0, n, 1 << 19):
        e = slice(s, min(n, s + (1 << 19)))
        xe, ce = x[e] - x[e][:, :1], c[e].double()
        for q, (w, ph, de) in enumerate(zip(*rule)):
            ph = torch.tensor(ph, device=x.device, dtype=torch.float64)
            de = torch.tensor(de, device=x.device, dtype=torch.float64)
            J = torch.einsum("nrd,rj->ndj", xe, de)
            cof = torch.stack([torch.linalg.cross(J[..., 1], J[..., 2]), torch.linalg.cross(J[..., 2], J[..., 0]),
                               torch.linalg.cross(J[..., 0], J[..., 1])], 1)
            det = (J[..., 0] * cof[:, 0]).sum(-1)
            g = torch.einsum("rj,njd->nrd", de, cof) / det[:, None, None]
            vol = w * det.abs()
            cq = ce[:, q if case["mode"] == "point" else 0]
            if case["kind"] == "poisson":
                A[e] += vol[:, None, None] * (g @ g.mT)
                b[e] += (vol * cq[:, 0])[:, None] * ph
                continue
            P = torch.cat([ph[None, :, None].expand(len(g), ns, 1), g], 2)
            A[e] += vol[:, None, None] * (P @ cq[:, :16].reshape(-1, 4, 4) @ P.mT)
            b[e] += vol[:, None] * (P @ cq[:, 16:, None])[..., 0]
    return A, b


def exact(case, seed):
    if case["call"] == "batch":
        meshes = _meshes(case)
        offs, total = _offsets(meshes)
        out = [torch.zeros(k, device=_DEV, dtype=torch.float64) for k in total[:2]]
        for i, (c, o) in enumerate(zip(meshes, offs)):
            _, _, x, cf, _ = _inputs(c, seed * 1000 + i)
            for t, r, (a, b) in zip(out, _integrate_exact(c, x, cf), o):
                t[a:b] = r.reshape(-1)
        return out[0], out[1], None
    nodes, conn, x, c, gen = _inputs(case, seed)
    A, b = _integrate_exact(case, x, c)
    if case["call"] == "apply":
        v = _rand(gen, -1, 1, nodes.shape[0]).to(c.dtype).double()
        idx = conn.long()
        ye = (A @ v[idx][..., None])[..., 0]
        y = torch.zeros_like(v).index_add_(0, idx.reshape(-1), ye.reshape(-1))
        f = torch.zeros_like(v).index_add_(0, idx.reshape(-1), b.reshape(-1))
        return y, f
    if case["call"] == "integrate" and case["layout"] == "soa":
        return A.reshape(case["n"], -1).T.contiguous(), b.T.contiguous(), None
    return A, b, None
