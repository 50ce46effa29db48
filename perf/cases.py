"""What a user of this framework has it compute, as cases that can be timed and compared.

The framework is a fast-multipole boundary-element library for clusters of bubbles: operator
products of the single and the double layer (by the multipole method or directly), the build
that precedes them on every new geometry, Dirichlet solves, time steps and the learned initial
guess. Every case goes through the public binding (paper_1905_01341_gb300.bem). Sizes are those
of the repository's workloads (icospheres of levels 2 to 6, clusters of 1 to 5000 bubbles at a
mean spacing of four radii, 64 or fewer independent clusters) and sizes between them.

Every API vector is FP64. A program that runs the mixed-precision mode gets about seven digits
and keeps its results in single precision, so the mixed cases return float32 copies; the FP64
cases return the vectors as they are.
"""
import functools
import math

import numpy as np
import torch

from paper_1905_01341_gb300 import bem

DEV = "cuda"
INV4PI = 1.0 / (4.0 * math.pi)
MEAN_VERTS = {"2": 162, "3": 642, "4": 2562, "5": 10242, "6": 40962, "23": 402, "34": 1602, "234": 1122}
EXACT_N = 200000  # the direct 64-bit sums over more points take too long


def listed():
    return [
        # one bubble of 642 vertices, dense direct FP64 solve to 1e-10: the smallest whole call,
        # dominated by launches and host reads
        {"name": "solve_direct_642_fp64", "kind": "solve_direct", "bubbles": 1, "levels": "3", "precision": "fp64"},
        # the allocation-free direct product of a latency-critical loop, an odd number of points
        {"name": "direct_noalloc_13446", "kind": "noalloc", "bubbles": 3, "levels": "534", "op": "both"},
        # a single finely meshed bubble (40962 vertices), one single-layer product
        {"name": "sl_bubble_40962", "kind": "apply", "bubbles": 1, "levels": "6", "op": "sl", "precision": "mixed", "p": 14},
        # the FP64-accuracy path on a single bubble, both layers at once
        {"name": "both_bubble_40962_fp64", "kind": "apply", "bubbles": 1, "levels": "6", "op": "both", "precision": "fp64", "p": 16},
        # the product of every solver iteration on an ordinary cluster
        {"name": "sl_cluster_300", "kind": "apply", "bubbles": 300, "levels": "3", "op": "sl", "precision": "mixed", "p": 14},
        # ... and on the largest one (3.21M unknowns)
        {"name": "sl_cluster_5000", "kind": "apply", "bubbles": 5000, "levels": "3", "op": "sl", "precision": "mixed", "p": 14},
        # the right-hand side of a solve (double layer) on bubbles meshed unevenly
        {"name": "rhs_cluster_500_uneven", "kind": "apply", "bubbles": 500, "levels": "34", "op": "rhs", "precision": "mixed", "p": 14},
        # new vertex positions: geometry, octree, lists and the singular diagonals (four right-hand
        # sides), done once per time-step stage
        {"name": "build_cluster_1500", "kind": "build", "bubbles": 1500, "levels": "3", "precision": "mixed", "p": 14},
        # a Dirichlet solve to 1e-6 with the bubble-block preconditioner
        {"name": "solve_cluster_100_uneven", "kind": "solve", "bubbles": 100, "levels": "34", "precision": "mixed", "p": 14},
        # one Adams-Bashforth step of a cluster in an acoustic field
        {"name": "step_cluster_300", "kind": "step", "bubbles": 300, "levels": "3", "clusters": 1, "p": 14},
        # independent clusters of uneven size stepped together
        {"name": "step_batched_16", "kind": "step", "bubbles": 320, "levels": "234", "clusters": 16, "p": 14},
        # a training batch of the learned initial guess (1000 bubbles' coefficients)
        {"name": "mlp_grad_1000", "kind": "mlp", "batch": 1000, "hidden": 256, "lmax": 10, "op": "grad"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve_direct", "noalloc", "direct", "apply", "apply", "apply", "apply64", "build", "solve", "step",
                       "batched", "mlp"])
    if kind == "solve_direct":
        return {"kind": kind, "bubbles": rng.randint(1, 3), "levels": rng.choice(["2", "3", "23"]),
                "precision": rng.choice(["fp64", "mixed"])}
    if kind in ("noalloc", "direct"):
        levels = rng.choice(["2", "3", "4", "23", "34"])
        nb = max(1, _log_int(rng, 162, 20000) // MEAN_VERTS[levels])
        case = {"kind": "noalloc", "bubbles": nb, "levels": levels, "op": rng.choice(["sl", "dl", "both"])}
        if kind == "direct":
            case = {**case, "kind": "direct", "precision": rng.choice(["fp64", "mixed"])}
        return case
    if kind == "apply64":
        levels = rng.choice(["3", "4", "34"])
        nb = max(1, _log_int(rng, 2000, 40000) // MEAN_VERTS[levels])
        return {"kind": "apply", "bubbles": nb, "levels": levels, "op": rng.choice(["sl", "dl", "both", "rhs"]),
                "precision": "fp64", "p": rng.choice([12, 16])}
    levels = rng.choice(["3", "4", "34", "234"])
    if kind == "apply":
        nb = max(1, _log_int(rng, 2000, 2000000) // MEAN_VERTS[levels])
        return {"kind": kind, "bubbles": nb, "levels": levels, "op": rng.choice(["sl", "sl", "sl", "dl", "both", "rhs"]),
                "precision": "mixed", "p": rng.choice([8, 10, 12, 13, 14, 14, 14, 16])}
    if kind == "build":
        nb = max(1, _log_int(rng, 2000, 900000) // MEAN_VERTS[levels])
        return {"kind": kind, "bubbles": nb, "levels": levels, "precision": "mixed", "p": rng.choice([10, 12, 14, 14])}
    if kind == "solve":
        nb = max(1, _log_int(rng, 2000, 150000) // MEAN_VERTS[levels])
        return {"kind": kind, "bubbles": nb, "levels": levels, "precision": "mixed", "p": 14}
    if kind == "step":
        nb = max(1, _log_int(rng, 2000, 180000) // MEAN_VERTS[levels])
        return {"kind": kind, "bubbles": nb, "levels": levels, "clusters": 1, "p": rng.choice([12, 14])}
    if kind == "batched":
        clusters = rng.randint(2, 16)
        return {"kind": "step", "bubbles": clusters * rng.randint(2, 19), "levels": "234", "clusters": clusters, "p": 14}
    return {"kind": "mlp", "batch": _log_int(rng, 16, 4000), "hidden": 16 * rng.randint(2, 16), "lmax": rng.randint(4, 10),
            "op": rng.choice(["grad", "grad", "forward"])}


# ------------------------------------------------------------------------------------ inputs


@functools.lru_cache(maxsize=None)
def _icosphere(level):
    """Unit icosphere: 10 * 4^level + 2 vertices, counter-clockwise triangles seen from outside."""
    t = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    f = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                  (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11),
                  (6, 2, 10), (8, 6, 7), (9, 8, 1)])
    for _ in range(level):
        e = np.sort(np.stack([f, np.roll(f, -1, axis=1)], axis=2).reshape(-1, 2), axis=1)
        uniq, inv = np.unique(e, axis=0, return_inverse=True)
        mid = v[uniq[:, 0]] + v[uniq[:, 1]]
        m = (len(v) + inv.reshape(-1, 3))
        v = np.concatenate([v, mid / np.linalg.norm(mid, axis=1, keepdims=True)])
        ab, bc, ca = m[:, 0], m[:, 1], m[:, 2]
        f = np.concatenate([np.stack(c, axis=1) for c in ((f[:, 0], ab, ca), (f[:, 1], bc, ab), (f[:, 2], ca, bc),
                                                          (ab, bc, ca))])
    return v, f.astype(np.int32)


def _place(radii, rng):
    """Centres uniform in a cube of side 4 M^(1/3), surfaces at least half the larger radius apart;
    the largest bubbles first."""
    m = len(radii)
    box = max(4.0 * m ** (1.0 / 3.0), 2.0 * float(radii.max()))
    placed, r_placed, centres = np.empty((m, 3)), np.empty(m), np.empty((m, 3))
    for k, i in enumerate(np.argsort(-radii, kind="stable")):
        need2 = (r_placed[:k] + radii[i] + 0.5 * np.maximum(r_placed[:k], radii[i])) ** 2
        for tries in range(100000):
            if tries % 200 == 199:
                box *= 1.05  # a crowded small cluster
            c = (rng.random(3) - 0.5) * box
            d = placed[:k] - c
            if not np.any((d * d).sum(axis=1) < need2):
                break
        placed[k], r_placed[k], centres[i] = c, radii[i], c
    return centres


def _mesh(case, seed):
    """Vertices [N, 3], triangles [T, 3], offsets, per-vertex bubble and direction, radii, clusters."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nb, clusters = case["bubbles"], case.get("clusters", 1)
    radii = np.exp(0.3 * rng.standard_normal(nb)) if nb > 1 else np.ones(1)
    # uneven clusters: at least one bubble each, the rest at random
    boff = np.concatenate([[0], np.sort(rng.choice(np.arange(1, nb), clusters - 1, replace=False)), [nb]]).astype(np.int64)
    centres = np.concatenate([_place(radii[a:b], rng) for a, b in zip(boff[:-1], boff[1:])])
    digits = [int(d) for d in case["levels"]]
    levels = np.resize(digits, nb)  # every level equally often: the size does not depend on the seed
    levels = levels if nb == len(digits) else rng.permutation(levels)
    deform = case["kind"] not in ("step",)  # a time integration starts from spheres
    xs, ts, us, voff, toff = [], [], [], [0], [0]
    for r, c, lev in zip(radii, centres, levels):
        u, f = _icosphere(int(lev))
        rad = r
        if deform:
            a = rng.standard_normal(3)
            z = u @ (a / np.linalg.norm(a))
            rad = (r * (1.0 + 0.05 * rng.standard_normal() * (1.5 * z * z - 0.5)))[:, None]
        xs.append(u * rad + c)
        us.append(u)
        ts.append(f + voff[-1])
        voff.append(voff[-1] + len(u))
        toff.append(toff[-1] + len(f))
    voff, toff = np.array(voff, np.int64), np.array(toff, np.int64)
    return {"xyz": torch.from_numpy(np.concatenate(xs)).to(DEV), "tri": torch.from_numpy(np.concatenate(ts)).to(DEV),
            "u": torch.from_numpy(np.concatenate(us)).to(DEV), "voff": voff, "toff": toff, "boff": boff,
            "radii": torch.from_numpy(radii).to(DEV),
            "bub": torch.repeat_interleave(torch.arange(nb, device=DEV), torch.from_numpy(np.diff(voff)).to(DEV))}


def _smooth(m, seed, lmax=6):
    """Per bubble a random series of Legendre polynomials P_l(u . e_l), l <= lmax, times 0.01 R."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    nb, b = len(m["radii"]), m["bub"]
    out = torch.zeros(len(b), dtype=torch.float64, device=DEV)
    for l in range(lmax + 1):
        e = torch.randn(nb, 3, dtype=torch.float64, device=DEV, generator=g)
        e /= e.norm(dim=1, keepdim=True)
        coef = torch.randn(nb, dtype=torch.float64, device=DEV, generator=g) * (0.01 * (2 * l + 1) * math.sqrt(INV4PI)) * m["radii"]
        x = (m["u"] * e[b]).sum(dim=1)
        p0, p1 = torch.ones_like(x), x
        for n in range(1, l):
            p0, p1 = p1, ((2 * n + 1) * x * p1 - n * p0) / (n + 1)
        out += coef[b] * (p0 if l == 0 else p1)
    return out


def _density(m, seed):
    """A solver's vector: a smooth part and a rough one."""
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    s = _smooth(m, seed + 2)
    return s + 0.3 * float(s.std()) * torch.randn(len(s), dtype=torch.float64, device=DEV, generator=g)


def _context(m, **params):
    ctx = bem.BemContext(**params)
    ctx.upload(m["xyz"].T.contiguous(), m["tri"].T.contiguous(), m["voff"], m["toff"])
    if len(m["boff"]) > 2:
        bem.bem_mesh_set_clusters(ctx.ctx, len(m["boff"]) - 1, m["boff"])
    return ctx


FG = {"sl": (1.0, 0.0), "dl": (0.0, 1.0), "both": (1.0, -0.5)}


def _mlp_inputs(case, seed):
    """Features (roughly unit columns, as after scaling), targets and He-initialised parameters."""
    psh = (case["lmax"] + 1) ** 2
    dims = [3 * psh, case["hidden"], case["hidden"], case["hidden"], psh]
    g = torch.Generator(device=DEV).manual_seed(seed)
    rnd = lambda *s: torch.randn(*s, dtype=torch.float64, device=DEV, generator=g)  # noqa: E731
    F, T = rnd(case["batch"], dims[0]), rnd(case["batch"], dims[4])
    parts = []
    for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        parts += [rnd(b * a) * math.sqrt(2.0 / a) * (0.1 if i == 3 else 1.0), 0.05 * rnd(b)]
    return dims, F, T, torch.cat(parts).float().double()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        m = _mesh({"kind": "step", "bubbles": 1, "levels": "3"}, seed)
        dims, F, T, params = _mlp_inputs(case, seed)
        ctx = _context(m, fixed_level=2)
        bem.bem_step_init(ctx.ctx, _smooth(m, seed))
        bem.bem_mlp_init(ctx.ctx, hidden=case["hidden"], lmax=case["lmax"])
        bem.bem_mlp_set_params(ctx.ctx, params)
        return {"case": case, "ctx": ctx, "F": F, "T": T, "grads": torch.empty_like(params),
                "Y": torch.empty(case["batch"], dims[4], dtype=torch.float64, device=DEV)}
    m = _mesh(case, seed)
    n = len(m["xyz"])
    prec = bem.BEM_PREC_FP64 if case.get("precision") == "fp64" else bem.BEM_PREC_MIXED
    st = {"case": case, "out": torch.empty(n, dtype=torch.float64, device=DEV), "n": n}
    if kind in ("solve_direct", "direct", "noalloc"):
        ctx = _context(m, mvp=bem.BEM_MVP_DIRECT, precision=prec, gmres_tol=1e-10 if case.get("precision") == "fp64" else 1e-6)
    elif kind == "step":
        ctx = _context(m, precision=bem.BEM_PREC_MIXED, p_fmm=case["p"], gmres_precond=2)
    else:
        ctx = _context(m, precision=prec, p_fmm=case["p"], gmres_precond=2 if kind == "solve" else 0)
    st["ctx"] = ctx
    if kind == "step":
        # past the Runge-Kutta start; each pass steps from the state reached here, its solve
        # starting from the solution one step before
        sp = bem.bem_step_params_default(pa=0.5, guess=0)
        bem.bem_step_init(ctx.ctx, _smooth(m, seed), sp)
        e = lambda *s: torch.empty(*s, dtype=torch.float64, device=DEV)  # noqa: E731
        st["from"], st["to"] = [[e(3, n), e(n), e(n)] for _ in range(2)]
        for k in range(5):
            bem.bem_step_get_state(ctx.ctx, q=st["from"][2])
            bem.bem_step(ctx.ctx)
        bem.bem_step_get_state(ctx.ctx, *st["from"][:2])
        return st
    if kind == "build":
        st["xyz"] = m["xyz"].T.contiguous()
        st["geo"] = [torch.empty(k, dtype=torch.float64, device=DEV) for k in (n, 3 * n, n, n)]
        return st
    ctx.build()
    st["xL"], st["xM"] = _density(m, seed), _smooth(m, seed + 3, lmax=8)
    if kind in ("solve", "solve_direct"):
        st["q0"] = torch.zeros(n, dtype=torch.float64, device=DEV)
        if kind == "solve":  # the preconditioner is kept over the solves that follow
            bem.bem_precond_apply(ctx.ctx, st["xM"], st["out"])
    if kind == "noalloc":
        st["xyz"] = m["xyz"].T.contiguous()
        st["geo"] = [torch.empty(k, dtype=torch.float64, device=DEV) for k in (n, 3 * n, n, n)]
        bem.bem_get_geometry(ctx.ctx, *st["geo"])
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "mlp":
        if case["op"] == "forward":
            bem.bem_mlp_forward(ctx.ctx, st["F"], st["Y"])
            return {"Y": st["Y"].float()}
        loss = bem.bem_mlp_loss_grad(ctx.ctx, st["F"], st["T"], st["grads"])
        return {"loss": loss, "grads": st["grads"].float()}
    if kind == "step":
        bem.bem_step_set_state(ctx.ctx, *st["from"])
        bem.bem_step(ctx.ctx)
        bem.bem_step_get_state(ctx.ctx, *st["to"])
        return {k: v.float() for k, v in zip(("xyz", "phi", "q"), st["to"])}
    single = case.get("precision") != "fp64"
    if kind == "build":
        bem.bem_mesh_update_xyz(ctx.ctx, st["xyz"])
        ctx.build()
        s, n, ld, md = st["geo"]
        bem.bem_get_geometry(ctx.ctx, s, n, ld, md)
        return {"s": s, "n": n, "ldiag": ld.float() if single else ld, "mdiag": md.float() if single else md}
    out = st["out"]
    if kind in ("solve", "solve_direct"):
        out.copy_(st["q0"])
        ctx.solve(st["xM"], out)
    elif kind == "noalloc":
        f, g = FG[case["op"]]
        s, n, ld, md = st["geo"]
        bem.bem_apply_direct_noalloc(st["n"], st["xyz"], s, n, ld, md, f, st["xL"], g, st["xM"], out,
                                     torch.cuda.current_stream())
    elif case["op"] == "rhs":
        bem.bem_rhs(ctx.ctx, st["xM"], out)
    else:
        f, g = FG[case["op"]]
        ctx.apply(f, st["xL"], g, st["xM"], out)
    return out.float() if single else out


# ------------------------------------------------------------------------------------ work


def work(case):
    """Inputs read once and outputs written once; operations: 11 per pair of a single layer and 19 of
    a double layer, over all pairs of a direct product, over about 800 near pairs a point of a
    multipole product (13 leaves of 64 points on a surface) plus 4 p^2 a point for its expansions at
    the leaves (what the translations cost depends on the scheme: not counted)."""
    kind = case["kind"]
    if kind == "mlp":
        psh = (case["lmax"] + 1) ** 2
        dims = [3 * psh, case["hidden"], case["hidden"], case["hidden"], psh]
        par = sum(a * b + b for a, b in zip(dims[:-1], dims[1:]))
        passes = 3 if case["op"] == "grad" else 1
        out = par if case["op"] == "grad" else case["batch"] * psh
        return {"bytes": 8.0 * (case["batch"] * (dims[0] + (psh if passes == 3 else 0)) + out) + 2.0 * par,
                "flops": 2.0 * passes * case["batch"] * par}
    n = float(sum(MEAN_VERTS[d] for d in (case["levels"] * case["bubbles"])[:case["bubbles"]]))
    per = {"sl": 11, "dl": 19, "rhs": 19, "both": 30}.get(case.get("op"), 11)
    if kind in ("direct", "noalloc"):
        return {"bytes": 8 * n * 12, "flops": n * n * per}
    if kind == "solve_direct":  # about 20 products, and 4 vectors in and out
        return {"bytes": 8 * n * 10, "flops": 20 * n * n * 11}
    near = 800 * n
    ends = 4 * case["p"] ** 2 * n
    if kind == "apply":
        return {"bytes": 8 * n * 12, "flops": near * per + ends}
    build = near * 33 + 4 * ends
    if kind == "build":
        return {"bytes": 8 * n * 15, "flops": build}
    solve = near * 19 + ends + 10 * (near * 11 + ends)  # about 10 products and the right-hand side
    if kind == "solve":
        return {"bytes": 8 * n * 10, "flops": solve}
    return {"bytes": 8 * n * 30, "flops": build + solve}


# ------------------------------------------------------------------------------------ 64-bit values


def _geometry(m):
    """Vertex weights (a third of the triangles' areas) and area-weighted unit normals."""
    x, t = m["xyz"], m["tri"].long()
    a = 0.5 * torch.linalg.cross(x[t[:, 1]] - x[t[:, 0]], x[t[:, 2]] - x[t[:, 0]])
    s, nrm = torch.zeros_like(x[:, 0]), torch.zeros_like(x)
    for c in range(3):
        s.index_add_(0, t[:, c], a.norm(dim=1) / 3.0)
        nrm.index_add_(0, t[:, c], a)
    return s, nrm / nrm.norm(dim=1, keepdim=True)


def _blocks(m, fn):
    """fn(rows, 1/r, 1/r^3) for all pairs by blocks of rows, zero where i = j."""
    x = m["xyz"] - m["xyz"].mean(dim=0)
    n = len(x)
    step = max(1, min(n, (1 << 27) // n))
    for a in range(0, n, step):
        r = slice(a, min(n, a + step))
        r2 = torch.zeros(r.stop - a, n, dtype=torch.float64, device=DEV)
        for d in range(3):
            r2 += (x[r, d, None] - x[None, :, d]) ** 2
        k = torch.arange(a, r.stop, device=DEV)
        r2[k - a, k] = math.inf
        ri = r2.rsqrt_()
        fn(r, x, ri, ri * ri * ri)


def _layers(m, xl, xm):
    """Off-diagonal L xl and M xm for columns xl [N, a], xm [N, b], and the identity diagonals."""
    s, nrm = _geometry(m)
    n, w = len(s), s * INV4PI
    x0 = m["xyz"] - m["xyz"].mean(dim=0)
    one = torch.ones(n, 1, dtype=torch.float64, device=DEV)
    A = torch.cat([xl, nrm], dim=1) * w[:, None]
    B = torch.cat([xm, one, x0], dim=1) * w[:, None]
    L, M = torch.empty_like(A), torch.empty_like(B)
    nx = (nrm * x0).sum(dim=1, keepdim=True)
    cols = torch.cat([B * nx] + [B * nrm[:, d:d + 1] for d in range(3)], dim=1)

    def part(r, x, ri, ri3):
        L[r] = ri @ A
        v = (ri3 @ cols).reshape(-1, 4, B.shape[1])
        M[r] = (x[r].T[:, :, None] * v[:, 1:].transpose(0, 1)).sum(dim=0) - v[:, 0]

    _blocks(m, part)
    a, b = xl.shape[1], xm.shape[1]
    md = -0.5 - M[:, b]
    ld = (nrm * (M[:, b + 1:b + 4] - L[:, a:a + 3] + (0.5 + md)[:, None] * x0)).sum(dim=1)
    return s, nrm, L[:, :a], M[:, :b], ld, md


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return None  # a time step of the whole method
    if kind == "mlp":
        dims, F, T, params = _mlp_inputs(case, seed)
        params.requires_grad_(case["op"] == "grad")
        h, off = F, 0
        for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
            W, c = params[off:off + a * b].reshape(b, a), params[off + a * b:off + a * b + b]
            off += a * b + b
            h = h @ W.T + c
            h = h.relu() if i < 3 else h
        if case["op"] == "forward":
            return {"Y": h}
        loss = 0.5 * ((h - T) ** 2).sum() / len(F)
        return {"loss": float(loss), "grads": torch.autograd.grad(loss, params)[0]}
    m = _mesh(case, seed)
    n = len(m["xyz"])
    if kind == "build":
        if n > EXACT_N:
            s, nrm = _geometry(m)
            return {"s": s, "n": nrm.T.contiguous().reshape(-1), "ldiag": None, "mdiag": None}
        none = torch.empty(n, 0, dtype=torch.float64, device=DEV)
        s, nrm, _, _, ld, md = _layers(m, none, none)
        return {"s": s, "n": nrm.T.contiguous().reshape(-1), "ldiag": ld, "mdiag": md}
    if n > EXACT_N or (kind == "solve" and n > 20000):
        return None
    q, phi = _density(m, seed), _smooth(m, seed + 3, lmax=8)
    s, nrm, L, M, ld, md = _layers(m, q[:, None], phi[:, None])
    sl, dl = L[:, 0] + ld * q, M[:, 0] + md * phi
    if kind in ("solve", "solve_direct"):
        mat = torch.empty(n, n, dtype=torch.float64, device=DEV)

        def part(r, x, ri, ri3):
            mat[r] = ri * (s * INV4PI)

        _blocks(m, part)
        mat.diagonal().copy_(ld)
        return torch.linalg.solve(mat, dl - 0.5 * phi)
    if case["op"] == "rhs":
        return dl - 0.5 * phi
    f, g = FG[case["op"]]
    return f * sl + g * dl
