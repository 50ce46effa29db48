"""The kernels at the sizes where their tiling changes: tile remainders, groups of lanes, items cut
from long neighbour lists, split reductions, and both layouts of the tensor-core M2L.

Tolerances (relative L2): the bounds of the two paths, FP64 direct 1e-11 and mixed direct 2e-6
against the oracle, FP64 multipole products (p 17) 1e-6 and mixed ones (p 14) 1e-5; mixed against
FP64 at the same p (same truncation, arithmetic error only) 1e-5; solutions as products times the
conditioning, bounded by 50.
"""
import numpy as np
import pytest

import oracle
from oracle import mlp as omlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_mlp import _flatten, _unflatten, make_stepper, small_system  # noqa: E402
from test_gpu_parity import _bem, dev, make_ctx, rel, small_cluster  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1905_01341_gb300 import build

    build.build()


def product(ctx, f, xL, g, xM):
    o = torch.zeros(len(xL), dtype=torch.float64, device="cuda")
    ctx.apply(f, dev(xL), g, dev(xM), o)
    return o.cpu().numpy()


def densities(n, seed=12):
    rng = np.random.Generator(np.random.PCG64(seed))
    return rng.standard_normal(n), rng.standard_normal(n)


# 12, 42: below one warp of receivers; 132: just over 128; 1020 / 1032: around eight tiles of 128, one
# per block of a cluster; 84, 204: ragged tiles
@pytest.mark.parametrize("nb,level", [(1, 0), (1, 1), (2, 1), (11, 0), (17, 0), (85, 0), (86, 0)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (1, 2e-6)])
def test_direct_product_sizes(nb, level, prec, tol):
    mesh = small_cluster(nb, level, seed=5)
    ctx = make_ctx(mesh, mvp=_bem().BEM_MVP_DIRECT, precision=prec, diag_precision=0)
    ref = oracle.BemOperator(mesh.xyz, mesh.tri)
    xL, xM = densities(mesh.n)
    for f, g in ((1.0, 0.0), (0.0, 1.0), (0.7, -1.3)):
        assert rel(product(ctx, f, xL, g, xM), ref.apply(f, xL, g, xM)) < tol, (f, g)
    ctx.close()


# leaves of up to 8, 16, 32, 64 and more points: 8, 4, 2 and 1 groups of lanes, units and items cut
@pytest.mark.parametrize("leaf_target", [6, 12, 24, 48, 100, 300])
@pytest.mark.parametrize("prec,p,tol", [(0, 17, 1e-6), (1, 14, 1e-5)])
def test_multipole_product_leaf_sizes(leaf_target, prec, p, tol):
    mesh = small_cluster(20, 2, seed=11)
    ctx = make_ctx(mesh, mvp=_bem().BEM_MVP_FMM, precision=prec, p_fmm=p, leaf_target=leaf_target, diag_precision=0)
    ref = oracle.BemOperator(mesh.xyz, mesh.tri)
    xL, xM = densities(mesh.n)
    for f, g in ((1.0, 0.0), (0.0, 1.0), (0.7, -1.3)):
        assert rel(product(ctx, f, xL, g, xM), ref.apply(f, xL, g, xM)) < tol, (f, g)
    ctx.close()


# odd p: rows of p^2 floats that no 16-byte access fits; 16: the largest of the tensor-core M2L
@pytest.mark.parametrize("p", [4, 7, 10, 13, 15, 16])
def test_multipole_product_orders(p):
    mesh = small_cluster(20, 3, seed=11)
    xL, xM = densities(mesh.n)
    outs = {}
    for prec in (0, 1):
        ctx = make_ctx(mesh, mvp=_bem().BEM_MVP_FMM, precision=prec, p_fmm=p, leaf_target=32, diag_precision=0)
        outs[prec] = [product(ctx, f, xL, g, xM) for f, g in ((1.0, 0.0), (0.7, -1.3))]
        ctx.close()
    for a, b in zip(outs[1], outs[0]):
        assert rel(a, b) < 1e-5


# a sparse tree (a bubble's surface: pair-major rows) and a dense one (small bubbles filling a cube:
# target-major tiles), each against the pair-major and the CUDA-core form
@pytest.mark.parametrize("nb,bubble,level,dense", [(1, 4, 4, False), (1500, 1, 4, True), (800, 1, 3, True)])
@pytest.mark.parametrize("p", [8, 14, 16])
def test_m2l_layout_by_share_of_filled_rows(nb, bubble, level, dense, p):
    mesh = small_cluster(nb, bubble, seed=5)
    xL, xM = densities(mesh.n)
    outs = {}
    for key, prec, tc, tm in (("auto", 1, 1, 1), ("pair", 1, 1, 0), ("cc", 1, 0, 1), ("f64", 0, 0, 1)):
        ctx = make_ctx(mesh, mvp=_bem().BEM_MVP_FMM, precision=prec, p_fmm=p, fixed_level=level, m2l_tensor_cores=tc,
                       diag_precision=0, m2l_target_major=tm)
        outs[key] = product(ctx, 0.7, xL, -1.3, xM)
        ctx.close()
    # the layout is seen by its sums: the same rows give the same bits, other sums others
    assert np.array_equal(outs["auto"], outs["pair"]) != dense
    e = {k: rel(outs[k], outs["f64"]) for k in ("auto", "pair", "cc")}
    # pair-major rows are summed with compensation, as the CUDA-core form's; a target-major tile sums
    # its classes in the tensor cores' FP32 accumulators: the mixed path's bound
    assert e["auto"] < 1e-5 and e["pair"] < 2.0 * e["cc"] + 1e-7, e


# bubbles of one shape around 128 (the block preconditioner's columns and its split of K), and
# unknowns of a few warps up to several blocks of the fused Arnoldi step
@pytest.mark.parametrize("nb,level", [(2, 0), (12, 1), (129, 0), (130, 1), (9, 3)])
def test_preconditioned_solve_sizes(nb, level):
    bem = _bem()
    mesh = small_cluster(nb, level, seed=3)
    phi = 1.0 + 0.1 * densities(mesh.n)[0]
    qs = {}
    for prec, tol in ((0, 1e-10), (1, 1e-7)):
        ctx = make_ctx(mesh, mvp=bem.BEM_MVP_DIRECT, precision=prec, gmres_tol=tol, gmres_maxit=400, gmres_restart=100,
                       gmres_precond=2)
        q = torch.zeros(mesh.n, dtype=torch.float64, device="cuda")
        _, rr = ctx.solve(dev(phi), q)
        assert rr <= tol
        qs[prec] = q.cpu().numpy()
        ctx.close()
    assert rel(qs[1], qs[0]) < 5e-4


# rows around the 128-row tile and around 512, where the products' K is split; widths that are no
# multiple of a tile
@pytest.mark.parametrize("batch", [1, 127, 129, 511, 512, 515])
@pytest.mark.parametrize("hidden,lmax", [(64, 3), (80, 5)])
def test_network_gradient_sizes(batch, hidden, lmax):
    bem = _bem()
    mesh, phi = small_system(2)
    ctx = make_stepper(mesh, phi, mvp=bem.BEM_MVP_DIRECT, precision=bem.BEM_PREC_FP64)
    bem.bem_mlp_init(ctx.ctx, hidden=hidden, lmax=lmax, seed=7)
    info = bem.bem_mlp_info(ctx.ctx)
    dims = info["dims"]
    flat = np.zeros(info["num_params"])
    bem.bem_mlp_get_params(ctx.ctx, flat)
    params = _unflatten(flat, dims)
    rng = np.random.Generator(np.random.PCG64(8))
    F = rng.standard_normal((batch, dims[0]))
    T = rng.standard_normal((batch, dims[4])) * 0.3
    Y, g = np.zeros((batch, dims[4])), np.zeros(info["num_params"])
    bem.bem_mlp_forward(ctx.ctx, F, Y)
    loss = bem.bem_mlp_loss_grad(ctx.ctx, F, T, g)
    Lref, gref = omlp.loss_and_grads_bf16(params, F, T)
    assert rel(Y, omlp.forward_bf16(params, F)[0]) < 1e-2
    assert abs(loss - Lref) < 1e-2 * Lref and rel(g, _flatten(gref)) < 1e-2
    ctx.close()
