"""Calls over their whole accepted range: no size is refused, answered with NaN, given scratch out of
proportion, or made to do its work twice, because of how a kernel lays out its blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_mlp import make_stepper, small_system  # noqa: E402
from test_gpu_parity import _bem  # noqa: E402


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
