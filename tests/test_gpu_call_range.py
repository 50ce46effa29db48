"""Calls over their whole accepted range: no size is refused, answered with NaN, given scratch out of
proportion, or made to do its work twice, because of how a kernel lays out its blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402
from test_gpu_mlp import make_stepper, small_system  # noqa: E402
from test_gpu_parity import _bem, dev, make_ctx, rel, small_cluster  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1905_01341_gb300 import build

    build.build()


def points(n, seed=1):
    rng = np.random.Generator(np.random.PCG64(seed))
    return torch.from_numpy(rng.random((3, n))).cuda()


def point_ctx(xyz, **params):
    bem = _bem()
    ctx = bem.BemContext(**params)
    bem.bem_points_upload(ctx.ctx, xyz.shape[1], xyz)
    ctx.build()
    return ctx


# 75 full blocks of receivers, and one receiver more: 608 blocks instead of 600, of the same length,
# all resident at once, so the times differ by a few per cent; a block that went over its sources a
# second time, after the others, would add at least a block's own time, more than half of the whole.
# The line lies between.
def test_direct_product_past_a_full_block_costs_no_second_pass():
    bem = _bem()
    runs = {}
    for n in (9600, 9601):
        ctx = point_ctx(points(n), mvp=bem.BEM_MVP_DIRECT, precision=bem.BEM_PREC_MIXED)
        x = torch.ones(n, dtype=torch.float64, device="cuda")
        runs[n] = (ctx, x, torch.empty_like(x))
    times = {n: [] for n in runs}
    for rep in range(9):
        for n, (ctx, x, out) in runs.items():
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            for _ in range(50):
                ctx.apply(1.0, x, 0.0, None, out)
            b.record()
            torch.cuda.synchronize()
            if rep:
                times[n].append(a.elapsed_time(b))
    for ctx, _, _ in runs.values():
        ctx.close()
    assert np.median(times[9601]) < 1.25 * np.median(times[9600]), times


# 65535 x 32 rows and one more. Every row's sums are formed alike in any batch, so a small batch of
# some of the rows gives the same bits; the loss against its definition on the network's own output,
# a mean of 2097121 FP32 terms summed by 128 blocks of 256 threads (their rounding is below 1e-5).
def test_network_takes_more_rows_than_a_grid_has_in_y():
    bem = _bem()
    mesh, phi = small_system(1)
    ctx = make_stepper(mesh, phi, mvp=bem.BEM_MVP_DIRECT, precision=bem.BEM_PREC_FP64)
    bem.bem_mlp_init(ctx.ctx, hidden=16, lmax=0, seed=7)
    info = bem.bem_mlp_info(ctx.ctx)
    d0, d4 = info["dims"][0], info["dims"][4]
    rows = 65535 * 32 + 1
    g = torch.Generator(device="cuda").manual_seed(3)
    F, T = (torch.randn(rows, d, dtype=torch.float64, device="cuda", generator=g) for d in (d0, d4))
    Y = torch.zeros(rows, d4, dtype=torch.float64, device="cuda")
    bem.bem_mlp_forward(ctx.ctx, F, Y)
    some = torch.tensor([0, 31, 32, 127, 128, rows // 2, rows - 34, rows - 33, rows - 2, rows - 1], device="cuda")
    Ys = torch.zeros(len(some), d4, dtype=torch.float64, device="cuda")
    bem.bem_mlp_forward(ctx.ctx, F[some].contiguous(), Ys)
    assert torch.equal(Y[some], Ys)
    grads = torch.zeros(info["num_params"], dtype=torch.float64, device="cuda")
    loss = bem.bem_mlp_loss_grad(ctx.ctx, F, T, grads)
    want = 0.5 * float(((Y - T.float()) ** 2).sum()) / rows
    assert abs(loss - want) < 1e-5 * want and bool(torch.isfinite(grads).all())
    ctx.close()


# Every box of level 4 with all its children at level 5, or with one of them at random: the levels above
# are the same, so the second tree has 4096 translations at the leaves where the first has 32768. FP64 is
# bound by its operations: 64 parents of a block that have 8 children on average in its octant instead of
# 64 need one of four groups of 16 columns, and the levels above (585 of 4681 full parents) stay, so the
# second takes about (0.25 x 4096 + 585) / 4681 = 0.34 of the first's time, and all of it when the columns
# without a child are multiplied too. The line lies between.
def test_translations_up_and_down_cost_what_the_children_are():
    bem = _bem()
    rng = np.random.Generator(np.random.PCG64(5))
    box = np.stack(np.meshgrid(*[np.arange(16)] * 3, indexing="ij"), -1).reshape(-1, 3)
    octs = np.stack(np.meshgrid(*[np.arange(2)] * 3, indexing="ij"), -1).reshape(-1, 3)
    ms = {}
    for name, child in (("all", np.broadcast_to(octs, (4096, 8, 3))), ("one", rng.integers(0, 2, (4096, 1, 3)))):
        x = ((box[:, None] + 0.25 + 0.5 * child) / 16.0).reshape(-1, 3)
        x = np.concatenate([x, [[0.0] * 3, [1.0] * 3]])  # the cube
        ctx = bem.BemContext(precision=bem.BEM_PREC_FP64, p_fmm=16, fixed_level=5, overlap=0)
        bem.bem_points_upload(ctx.ctx, len(x), torch.from_numpy(np.ascontiguousarray(x.T)).cuda())
        ctx.build()
        q = torch.ones(len(x), dtype=torch.float64, device="cuda")
        out = torch.empty_like(q)
        ctx.apply(1.0, q, 0.0, None, out)
        bem.bem_profile_enable(ctx.ctx)
        bem.bem_profile_read(ctx.ctx)
        for _ in range(5):
            ctx.apply(1.0, q, 0.0, None, out)
        prof = bem.bem_profile_read(ctx.ctx)
        ms[name] = np.array([prof["m2m"][0], prof["l2l"][0]])
        ctx.close()
    assert np.all(ms["one"] < 0.65 * ms["all"]), ms


# Trees whose lowest levels have one child per parent, in one octant for all (a tile's columns are then
# one octant's, in several passes) or in any: products of points (one right-hand side) against the sum
# over all pairs, and the diagonals of tiny bubbles (four) against the direct FP64 path. 1e-6: the bound
# of the FP64 multipole path at p >= 14.
@pytest.mark.parametrize("octants", ["one", "any"])
@pytest.mark.parametrize("p", [16, 17])
def test_one_child_per_parent_products(octants, p):
    bem = _bem()
    rng = np.random.Generator(np.random.PCG64(6))
    box = np.stack(np.meshgrid(*[np.arange(16)] * 3, indexing="ij"), -1).reshape(-1, 3)
    child = np.zeros((4096, 3)) if octants == "one" else rng.integers(0, 2, (4096, 3))
    x = np.concatenate([(box + 0.25 + 0.5 * child) / 16.0, [[0.0] * 3, [1.0] * 3]])
    q = torch.from_numpy(rng.random(len(x))).cuda()
    t = torch.from_numpy(x).cuda()
    inv = 1.0 / (t[:, None] - t[None]).norm(dim=2).fill_diagonal_(np.inf)
    ctx = bem.BemContext(precision=bem.BEM_PREC_FP64, p_fmm=p, fixed_level=6)
    bem.bem_points_upload(ctx.ctx, len(x), t.T.contiguous())
    ctx.build()
    out = torch.empty_like(q)
    ctx.apply(1.0, q, 0.0, None, out)
    assert rel(out.cpu(), (inv @ q / (4.0 * np.pi)).cpu()) < 1e-6
    ctx.close()


def test_one_child_per_parent_diagonals():
    bem = _bem()
    i = np.stack(np.meshgrid(np.arange(16), np.arange(16), np.arange(4), indexing="ij"), -1).reshape(-1, 3)
    centres = np.concatenate([(i + 0.3) / 16.0, [[0.0] * 3, [1.0] * 3]])
    mesh = synth.cluster(0, np.full(len(centres), 1e-3), centres)
    geo = []
    for par in ({"mvp": bem.BEM_MVP_DIRECT}, {"p_fmm": 17, "fixed_level": 6}):
        ctx = make_ctx(mesh, precision=bem.BEM_PREC_FP64, **par)
        d = [torch.empty(k * mesh.n, dtype=torch.float64, device="cuda") for k in (1, 3, 1, 1)]
        bem.bem_get_geometry(ctx.ctx, *d)
        out = torch.empty(mesh.n, dtype=torch.float64, device="cuda")
        ctx.apply(1.0, torch.ones_like(out), 0.5, torch.ones_like(out), out)
        geo.append([v.cpu() for v in (*d[2:], out)])
        ctx.close()
    for a, b in zip(*geo):
        assert rel(b, a) < 1e-6


# A sheet of 512 x 512 points, each in a leaf box of its own. What the first product may allocate, in bytes:
# strengths and potentials (4 N doubles), expansions of all boxes (two of p^2), a row of p^2 and the target-major
# index per translation, and the near field's sums, 8 receivers of 16 bytes per leaf for up to two items
# and an eighth more; 64 MB for the chunk tables and the rounding of 16 allocations. 64 slots per leaf and
# item would be 268 MB, not 75.
def test_near_field_scratch_of_small_leaves():
    bem = _bem()
    n, p = 512 * 512, 2
    g = (np.arange(512) + 0.5) / 512.0
    xy = np.stack(np.meshgrid(g, g, indexing="ij"), -1).reshape(-1, 2)
    xyz = torch.from_numpy(np.concatenate([xy, np.full((n, 1), 0.5)], axis=1).T.copy()).cuda()
    ctx = bem.BemContext(precision=bem.BEM_PREC_FP64, p_fmm=p, fixed_level=10)
    bem.bem_points_upload(ctx.ctx, n, xyz)
    ctx.build()
    st = ctx.stats()
    q = torch.ones(n, dtype=torch.float64, device="cuda")
    out = torch.empty_like(q)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx.apply(1.0, q, 0.0, None, out)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert st["leaves"] == n
    boxes = 2 * n + n // 3
    bound = 32 * n + 16 * p * p * boxes + (8 * p * p + 4) * st["m2l_pairs"] + 2 * 128 * n * 9 // 8 + (64 << 20)
    ctx.close()
    assert used < bound, (used, bound, st["m2l_pairs"])


# Orders whose FP32 M2L leaves the range of FP32 (19, 20, and 17, 18 through the diagonals' p + 2), beside
# the last ones that do not: mixed against FP64 at the same order (the same truncation), with the mixed
# path's bound 1e-5, the diagonals in FP64 and at the default, in the mixed precision.
@pytest.mark.parametrize("p", [15, 16, 17, 18, 19, 20])
@pytest.mark.parametrize("diag", [0, -1])
def test_mixed_products_of_high_order(p, diag):
    bem = _bem()
    mesh = small_cluster(20, 3, seed=11)
    rng = np.random.Generator(np.random.PCG64(12))
    xL, xM = dev(rng.standard_normal(mesh.n)), dev(rng.standard_normal(mesh.n))
    out = {}
    for prec in (0, 1):
        ctx = make_ctx(mesh, mvp=bem.BEM_MVP_FMM, precision=prec, p_fmm=p, leaf_target=32, diag_precision=diag)
        out[prec] = []
        for f, g in ((1.0, 0.0), (0.0, 1.0), (0.7, -1.3)):
            o = torch.zeros(mesh.n, dtype=torch.float64, device="cuda")
            ctx.apply(f, xL, g, xM, o)
            out[prec].append(o.cpu())
        ctx.close()
    for a, b in zip(out[1], out[0]):
        assert rel(a, b) < 1e-5


# The Arnoldi step by one cooperative kernel takes up to 2048 unknowns per SM, more by separate launches:
# cycles of a solve at either side of that line (full slices below it), in both precisions. A broken
# Arnoldi relation or a wrong column or rotation shows in a cycle's last estimate, which is the residual to
# rounding when all are right (r_0 - A d is evaluated with the same products; its own rounding is below
# 1e-7 of |b| in the mixed precision and 1e-13 in FP64).
@pytest.mark.parametrize("prec,p,slack", [(0, 6, 1e-12), (1, 8, 2e-7)])
def test_solves_either_side_of_the_fused_step(prec, p, slack):
    bem = _bem()
    limit = 2048 * torch.cuda.get_device_properties(0).multi_processor_count
    for nb in (limit // 642, limit // 642 + 1):
        r = int(np.ceil(nb ** (1.0 / 3.0)))
        centres = 4.0 * np.stack(np.meshgrid(*[np.arange(r)] * 3, indexing="ij"), -1).reshape(-1, 3)[:nb]
        mesh = synth.cluster(3, 0.6 + 0.8 * np.random.Generator(np.random.PCG64(4)).random(nb), centres)
        assert (mesh.n <= limit) == (nb == limit // 642)
        ctx = make_ctx(mesh, precision=prec, p_fmm=p, gmres_precond=1, gmres_restart=12, gmres_maxit=24, gmres_tol=1e-9)
        phi = dev(np.cos(mesh.xyz @ np.array([0.3, 0.2, 0.1])))
        q = torch.zeros(mesh.n, dtype=torch.float64, device="cuda")
        it, rr = ctx.solve(phi, q, raise_on_noconv=False)
        hist = bem.bem_get_residual_history(ctx.ctx)  # residual, 12 estimates, residual, 12 estimates, residual
        ctx.close()
        assert it == 24 and len(hist) == 27 and rr == hist[26] and bool(torch.isfinite(q).all())
        for e in (12, 25):
            assert abs(hist[e + 1] - hist[e]) <= slack + 1e-6 * hist[e], hist
            assert hist[e] < 0.5 * hist[e - 12], hist


# one cycle of 75 basis vectors (the residual falls by about 0.6 an iteration), FP64
def test_solve_with_more_than_64_basis_vectors():
    bem = _bem()
    mesh = small_cluster(12, 2, seed=3)
    ctx = make_ctx(mesh, mvp=bem.BEM_MVP_DIRECT, precision=bem.BEM_PREC_FP64, gmres_tol=1e-18, gmres_maxit=75)
    q = torch.zeros(mesh.n, dtype=torch.float64, device="cuda")
    phi = dev(1.0 + 0.1 * np.random.Generator(np.random.PCG64(4)).standard_normal(mesh.n))
    it, rr = ctx.solve(phi, q, raise_on_noconv=False)
    hist = np.array(bem.bem_get_residual_history(ctx.ctx))
    ctx.close()
    assert it == 75 and len(hist) == 77
    assert np.all(np.diff(hist[:76]) <= 0.0) and abs(hist[76] - hist[75]) < 1e-12 and rr < 1e-12


# A tree whose single-layer M2L takes the pair-major rows (p = 16: 1 KB a translation, 0.9 GB), on a device with
# less room than those: the target-major tiles take half as much. A first product allocates 1.0 GB with the
# rows and 0.5 GB with the tiles; 0.7 GB are left.
def test_product_without_room_for_pair_rows():
    bem = _bem()
    rng = np.random.Generator(np.random.PCG64(9))
    radii = np.exp(0.3 * rng.standard_normal(500))
    mesh = synth.cluster(np.resize([3, 4], 500), radii, synth._place_centres(radii, 4.0 * 500 ** (1 / 3), 0.5, rng))
    par = dict(precision=bem.BEM_PREC_MIXED, p_fmm=16, diag_precision=0)
    x = dev(rng.standard_normal(mesh.n))
    outs = []
    # every kernel is loaded before memory is short: both forms, the tiles on a dense tree
    warm = point_ctx(points(100000), **par)
    warm.apply(1.0, torch.ones(100000, dtype=torch.float64, device="cuda"), 0.0, None,
               torch.empty(100000, dtype=torch.float64, device="cuda"))
    warm.close()
    for short in (False, True):
        ctx = make_ctx(mesh, **par)
        pairs = ctx.stats()["m2l_pairs"]
        out = torch.empty_like(x)
        torch.cuda.empty_cache()
        fill = None
        if short:
            assert 1024 * pairs > 700 << 20  # the rows alone have no room
            free = torch.cuda.mem_get_info()[0]
            fill = torch.empty(free - (700 << 20), dtype=torch.uint8, device="cuda")
        try:
            ctx.apply(1.0, x, 0.0, None, out)
            ctx.apply(1.0, x, 0.0, None, out)
            outs.append(out.cpu().numpy())
        finally:
            del fill
            ctx.close()
            torch.cuda.empty_cache()
    # other sums of the same translations: the mixed path's bound, and not the same bits
    assert 0.0 < rel(outs[1], outs[0]) < 1e-5


# 3 x 8 bytes of a million points have no room in 8 MB; once there is room, the next calls work.
def test_calls_after_a_refused_allocation():
    bem = _bem()
    xyz = points(1000000)
    q = torch.ones(xyz.shape[1], dtype=torch.float64, device="cuda")
    out = torch.empty_like(q)
    ctx = bem.BemContext(p_fmm=8)
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (8 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(bem.BemError) as ei:
            bem.bem_points_upload(ctx.ctx, xyz.shape[1], xyz)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert ei.value.code == bem.BEM_ERR_NOMEM
    bem.bem_points_upload(ctx.ctx, xyz.shape[1], xyz)
    ctx.build()
    ctx.apply(1.0, q, 0.0, None, out)
    assert bool(torch.isfinite(out).all())
    ctx.close()
