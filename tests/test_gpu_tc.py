"""Tensor-core (BF16 / FP16 operand) aggregation through the C ABI.

Tolerances come from the arithmetic: with unit roundoff u of the 16-bit type
(2^-9 for BF16, 2^-11 for FP16) applied to every cost and every weight, and
the normaliser summed from the same rounded weights in FP32,
    |Agg_tc - Agg| <= u max|C| + 2u max|C - Agg| / (1 - u) + FP32 terms
                   <= 3 u R + 1e-5          (R = cost range = 2 for NCC).
"""

import numpy as np
import pytest

from tests._compare import check_disparities, near_tie_mask

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = {"bf16": 2.0 ** -9, "f16": 2.0 ** -11}


@pytest.fixture(scope="module")
def fbs():
    from paper_1807_02044_gb300 import build as b
    b.build()
    import paper_1807_02044_gb300 as m
    return m


def _prec(fbs, name):
    return fbs.FBS_PREC_BF16 if name == "bf16" else fbs.FBS_PREC_F16


def _round16(a, name):
    t = torch.from_numpy(np.ascontiguousarray(a, np.float32))
    return (t.to(torch.bfloat16) if name == "bf16" else t.to(torch.float16)).to(torch.float32).numpy()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("H,W,D", [(8, 16, 16), (13, 37, 20), (24, 50, 64), (9, 40, 250), (10, 24, 256)])
def test_radius_zero_returns_the_rounded_cost_exactly(fbs, prec, H, W, D):
    """With radius 0 every pixel's only weight is 1, so the tensor-core product
    must reproduce the 16-bit cost bit for bit: this pins the operand layouts,
    the TMA box, the instruction descriptor and the accumulator read-out
    (D > 240: the two MMAs of N = 128 and N - 128 per K-step)."""
    rng = np.random.default_rng(H * W + D)
    cost = (rng.random((H, W, D)) * 2).astype(np.float32)
    G = rng.integers(0, 256, size=(H, W, 3)).astype(np.uint8)
    with fbs.Context(0, prec=_prec(fbs, prec)) as ctx:
        agg, di, ds = ctx.aggregate(_dev(cost), _dev(G), 0, 1.0, 10.0)
        torch.cuda.synchronize()
        fbs.fbs_sync(ctx.ctx)
    np.testing.assert_array_equal(agg.cpu().numpy(), _round16(cost, prec))


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("H,W,C,D,r", [(16, 24, 3, 16, 2), (21, 45, 3, 40, 7), (9, 70, 1, 64, 4), (30, 33, 3, 100, 9),
                                       (18, 300, 3, 256, 9), (11, 270, 1, 245, 5)])
def test_tc_aggregation_within_rounding_bound(fbs, oracle_mod, prec, H, W, C, D, r):
    rng = np.random.default_rng(7 * H + W)
    L = rng.integers(0, 256, size=(H, W, C)).astype(np.uint8)
    R = np.roll(L, -3, axis=1)
    with fbs.Context(0, prec=_prec(fbs, prec)) as ctx:
        dl, dr = _dev(L), _dev(R)
        cost = ctx.cost_volume(dl, dr, D)
        agg, di, ds = ctx.aggregate(cost, dl, r, float(r), 12.0)
        di2, ds2 = ctx.compute_disparity(dl, dr, D, r, float(r), 12.0)
        torch.cuda.synchronize()
        fbs.fbs_sync(ctx.ctx)
    ref_di, ref_ds, ref_agg = oracle_mod.fbs(L, R, D, r, float(r), 12.0, want_agg=True)
    err = np.abs(agg.cpu().numpy() - ref_agg).max()
    tol = 3 * U[prec] * 2.0 + 1e-5
    assert err <= tol, f"max |dAgg| {err:.3e} > {tol:.3e}"
    # integer winners agree except where the oracle's two best are within 2*tol,
    # subpixel disparities within the rounding bound propagated through Eq. (10)
    di = di.cpu().numpy()
    ties = near_tie_mask(ref_agg, 2 * tol)
    assert np.all((di == ref_di) | ties)
    stats = check_disparities(di, ds.cpu().numpy(), ref_agg, ref_di, ref_ds, 2.0, tol=tol)
    print(f"{prec} {W}x{H} D={D} r={r}: max |dAgg| {err:.2e} (bound {tol:.2e}), {stats}")
    # the production entry point (16-bit cost built directly) agrees with the
    # debug route (FP32 cost rounded by the conversion kernel): same rounding
    assert np.array_equal(di, di2.cpu().numpy())
    np.testing.assert_allclose(ds.cpu().numpy(), ds2.cpu().numpy(), atol=1e-6)


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("H,W,C,D,r", [
    (26, 40, 3, 256, 24),   # one row a stage, two stages
    (21, 45, 1, 32, 16),    # the smallest radius that always takes two groups
    (20, 50, 3, 256, 9),    # two rows, two stages
    (33, 37, 1, 128, 15),   # two rows, three stages; odd counts of window rows in the border tiles
    (1, 5000, 1, 256, 12),  # one stage a tile, several tiles a block: the groups take whole tiles in turn
])
def test_tc_two_producer_groups(fbs, oracle_mod, prec, H, W, C, D, r):
    """Shapes whose stages two groups of producer warps write in turn: the same
    bound as for every other shape."""
    test_tc_aggregation_within_rounding_bound(fbs, oracle_mod, prec, H, W, C, D, r)


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("D", [1, 2, 15, 16, 17, 31, 32, 33, 48, 100, 240, 241, 256])
def test_tc_winner_takes_the_first_of_equal_costs(fbs, prec, D):
    """With radius 0 the aggregated value is the cost itself.  Costs of four
    values only: every pixel has ties within and across the blocks of 16 that the
    epilogue reads, and winners at their edges; maps exactly the first minimum and
    its parabola in FP32."""
    H, W = 19, 37
    rng = np.random.default_rng(D)
    cost = (rng.integers(0, 4, size=(H, W, D)) / 8 + 0.25).astype(np.float32)
    cost[:8] += 0.25                             # upper rows: a single smallest value
    np.put_along_axis(cost[:8], rng.integers(0, D, size=(8, W, 1)), np.float32(0.125), axis=2)
    guide = rng.integers(0, 256, size=(H, W, 3)).astype(np.uint8)
    with fbs.Context(0, prec=_prec(fbs, prec)) as ctx:
        _, di, ds = ctx.aggregate(_dev(cost), _dev(guide), 0, 1.0, 12.0)
        torch.cuda.synchronize()
        fbs.fbs_sync(ctx.ctx)
    k = cost.argmin(axis=2)
    np.testing.assert_array_equal(di.cpu().numpy(), k)
    pad = np.pad(cost, ((0, 0), (0, 0), (1, 1)))
    at = [np.take_along_axis(pad, (k + i)[..., None], axis=2)[..., 0] for i in (0, 1, 2)]
    dd = 2 * at[0] + 2 * at[2] - 4 * at[1]
    inner = (k > 0) & (k < D - 1) & (dd > 0)
    ref = np.where(inner, k + (at[0] - at[2]) / np.where(inner, dd, 1), k).astype(np.float32)
    np.testing.assert_array_equal(ds.cpu().numpy(), ref)


@pytest.mark.parametrize("D", [16, 23, 40, 256])
def test_tc_winner_at_every_place(fbs, D):
    """With radius 0 the aggregated value is the cost itself (16ths up to 8, exact in 16 bits).  Pixel x of a row has
    its smallest cost at d = x: alone; with an equal one next to it; with one further on; after costs that fall to
    it from place to place; among far larger ones.  Winner and parabola (Eq. (10)) as in FP32."""
    rng = np.random.default_rng(D)
    A = (rng.integers(32, 129, (5, D, D)) / 16).astype(np.float32)
    x = np.arange(D)
    for d in range(D):
        A[3, d, :d + 1] = 1.0 + np.minimum(7.0, (d - x[:d + 1]) / 16)
        A[4, d, rng.random(D) < 0.5] = 512.0
        if d + 1 < D:
            A[1, d, d + 1] = 1.0
            A[2, d, rng.integers(d + 1, D)] = 1.0
    A[:, x, x] = 1.0
    assert np.array_equal(A.argmin(2), np.broadcast_to(x, (5, D)))
    cost, guide = torch.from_numpy(A).cuda(), torch.zeros((5, D, 3), dtype=torch.uint8, device="cuda")
    with fbs.Context(0, prec=fbs.FBS_PREC_F16) as ctx:
        _, di, ds = ctx.aggregate(cost, guide, 0, 1.0, 10.0)
        torch.cuda.synchronize()
        fbs.fbs_sync(ctx.ctx)
    assert np.array_equal(di.cpu().numpy(), np.broadcast_to(x, (5, D)))
    i = x[1:-1]
    a, b, c = A[:, i, i - 1], A[:, i, i], A[:, i, i + 1]
    den = np.float32(2) * a + np.float32(2) * c - np.float32(4) * b
    sub = i + np.where(den > 0, (a - c) / np.where(den > 0, den, np.float32(1)), np.float32(0))
    got = ds.cpu().numpy()
    assert np.array_equal(got[:, [0, -1]], np.broadcast_to(x[[0, -1]], (5, 2)).astype(np.float32))
    np.testing.assert_allclose(got[:, 1:-1], sub.astype(np.float32), rtol=0, atol=2.0 ** -22 * D)


@pytest.mark.parametrize("prec", ["bf16", "f16"])
def test_tc_full_size_bench_workload_bad_pixels(fbs, oracle_mod, prec):
    """640x480 RGB, D=64, radius 7 (the benchmark workload): aggregated costs
    of 400 sampled pixels within the 16-bit rounding bound of the FP64 oracle
    (the largest error is printed), their integer and subpixel disparities
    under the 16-bit rules, and extra bad pixels (> 1 px) of the 16-bit form
    over the FP32 form at most 0.5% on the sample and on the whole frame."""
    from synth import make_pair
    p = make_pair("rgb640x480_d64_r7", 0)
    dl, dr = _dev(p.left), _dev(p.right)
    out = {}
    for name, pr in [("f32", fbs.FBS_PREC_F32), (prec, _prec(fbs, prec))]:
        with fbs.Context(0, prec=pr) as ctx:
            di, ds = ctx.compute_disparity(dl, dr, p.D, p.radius, p.sigma_s, p.sigma_r, p.tau)
            torch.cuda.synchronize()
            fbs.fbs_sync(ctx.ctx)
            out[name] = (di.cpu().numpy(), ds.cpu().numpy())
    # the aggregated volume of the 16-bit form (debug route: the FP32 cost
    # rounded by the conversion kernel, the same rounding as the cost kernel)
    with fbs.Context(0, prec=_prec(fbs, prec)) as ctx:
        cost = ctx.cost_volume(dl, dr, p.D)
        agg, adi, ads = ctx.aggregate(cost, dl, p.radius, p.sigma_s, p.sigma_r)
        torch.cuda.synchronize()
        fbs.fbs_sync(ctx.ctx)
    assert np.array_equal(adi.cpu().numpy(), out[prec][0])
    rng = np.random.default_rng(1)
    ys = rng.integers(0, p.H, 400)
    xs = rng.integers(0, p.W, 400)
    ref_di, ref_ds, ref_agg = oracle_mod.fbs_points(p.left, p.right, p.D, p.radius, p.sigma_s, p.sigma_r, xs, ys)
    agg_s = agg[torch.from_numpy(ys).cuda(), torch.from_numpy(xs).cuda()].cpu().numpy()
    err = float(np.abs(agg_s - ref_agg).max())
    tol = 3 * U[prec] * 2.0 + 1e-5
    stats = check_disparities(out[prec][0][ys, xs], out[prec][1][ys, xs], ref_agg, ref_di, ref_ds, 2.0, tol=tol)
    print(f"640x480 D=64 r=7 {prec}: max |dAgg| vs FP64 oracle {err:.3e} (bound {tol:.3e}); {stats}")
    assert err <= tol
    bad32 = np.mean(np.abs(out["f32"][1][ys, xs] - ref_ds) > 1.0)
    bad16 = np.mean(np.abs(out[prec][1][ys, xs] - ref_ds) > 1.0)
    assert bad16 - bad32 <= 0.005, (bad32, bad16)
    # whole frame against the FP32 path
    whole = float(np.mean(np.abs(out[prec][1] - out["f32"][1]) > 1.0))
    print(f"640x480 D=64 r=7 {prec}: extra bad pixels over FP32 {100 * whole:.4f}%")
    assert whole <= 0.005


def test_tc_f16_1280x960_d128_r15(fbs, oracle_mod):
    """The precision-at-scale workload: 1280x960 RGB, D=128, radius 15, FP16
    operands.  Sampled aggregated costs within the FP16 rounding bound of the
    FP64 oracle; extra bad pixels (> 1 px) over the FP32 form at most 0.5%."""
    from synth import make_pair
    p = make_pair("rgb1280x960_d128_r15", 0)
    dl, dr = _dev(p.left), _dev(p.right)
    with fbs.Context(0, prec=fbs.FBS_PREC_F32) as c32:
        _, ds32 = c32.compute_disparity(dl, dr, p.D, p.radius, p.sigma_s, p.sigma_r)
        torch.cuda.synchronize()
    with fbs.Context(0, prec=fbs.FBS_PREC_F16) as c16:
        di16, ds16 = c16.compute_disparity(dl, dr, p.D, p.radius, p.sigma_s, p.sigma_r)
        cost = c16.cost_volume(dl, dr, p.D)
        agg, _, _ = c16.aggregate(cost, dl, p.radius, p.sigma_s, p.sigma_r)
        torch.cuda.synchronize()
        fbs.fbs_sync(c16.ctx)
    rng = np.random.default_rng(9)
    xs, ys = rng.integers(0, p.W, 60), rng.integers(0, p.H, 60)
    ref_di, ref_ds, ref_agg = oracle_mod.fbs_points(p.left, p.right, p.D, p.radius, p.sigma_s, p.sigma_r, xs, ys)
    agg_s = agg[torch.from_numpy(ys).cuda(), torch.from_numpy(xs).cuda()].cpu().numpy()
    err = np.abs(agg_s - ref_agg).max()
    tol = 3 * U["f16"] * 2.0 + 1e-5
    stats = check_disparities(di16.cpu().numpy()[ys, xs], ds16.cpu().numpy()[ys, xs], ref_agg, ref_di, ref_ds, 2.0,
                              tol=tol)
    print(f"1280x960 D=128 r=15 FP16: max |dAgg| vs FP64 oracle {err:.3e} (bound {tol:.3e}); {stats}")
    assert err <= tol
    bad = float(np.mean(np.abs(ds16.cpu().numpy() - ds32.cpu().numpy()) > 1.0))
    print(f"extra bad pixels over FP32: {100 * bad:.4f}%")
    assert bad <= 0.005


@pytest.mark.parametrize("prec,expect", [("f32", {"COST": 2, "AGG_F32": 1, "AGG_TC": 0}),
                                         ("bf16", {"COST": 1, "AGG_F32": 0, "AGG_TC": 1})])
def test_kernel_accounting_counts_every_launch(fbs, prec, expect):
    """fbs_profile_read reports kernels, not calls: the FP32 form launches the
    statistics pre-pass, the cost kernel and the aggregation; the 16-bit form
    one cost kernel (statistics, pad rows and guide included) and the
    tensor-core aggregation."""
    rng = np.random.default_rng(3)
    L = rng.integers(0, 256, size=(40, 72, 3)).astype(np.uint8)
    R = np.roll(L, -2, axis=1)
    p = fbs.FBS_PREC_F32 if prec == "f32" else _prec(fbs, prec)
    with fbs.Context(0, prec=p) as ctx:
        dl, dr = _dev(L), _dev(R)
        ctx.compute_disparity(dl, dr, 24, 3, 3.0, 12.0)
        torch.cuda.synchronize()
        fbs.fbs_profile(ctx.ctx, 1)
        for _ in range(3):
            ctx.compute_disparity(dl, dr, 24, 3, 3.0, 12.0)
        torch.cuda.synchronize()
        got = {k: fbs.fbs_profile_read(ctx.ctx, getattr(fbs, "FBS_KERNEL_" + k))[1] for k in expect}
        fbs.fbs_profile(ctx.ctx, 0)
        fbs.fbs_sync(ctx.ctx)
    assert got == {k: 3 * v for k, v in expect.items()}



# The 16-bit cost kernel covers 64 pixels x 4 rows per CTA, 16 disparities per warp.
@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("H,W,C,D", [(1, 1, 1, 1), (3, 7, 3, 15), (4, 64, 1, 16), (5, 65, 3, 17), (9, 129, 3, 40),
                                     (6, 200, 1, 64), (2, 61, 3, 130), (7, 300, 3, 256)])
def test_radius_zero_maps_are_those_of_the_rounded_fp32_costs(fbs, prec, H, W, C, D):
    """With radius 0 the aggregated value is the 16-bit cost itself, so the maps are
    exactly those of the FP32 volume (another kernel) rounded to 16 bits."""
    rng = np.random.default_rng(H + W + D)
    L = rng.integers(0, 256, (H, W, C)).astype(np.uint8)
    R = np.roll(L, -min(5, W - 1), axis=1)
    R = np.clip(R.astype(np.int32) + rng.integers(-40, 41, R.shape), 0, 255).astype(np.uint8)
    L[:, : W // 3] //= 64                    # flat blocks and exact ties
    dl, dr = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
    with fbs.Context(0, prec=fbs.FBS_PREC_BF16 if prec == "bf16" else fbs.FBS_PREC_F16) as ctx:
        di, ds = ctx.compute_disparity(dl, dr, D, 0, 1.0, 10.0)
        cost = ctx.cost_volume(dl, dr, D)
        torch.cuda.synchronize()
        fbs.fbs_sync(ctx.ctx)
    A = cost.to(torch.bfloat16 if prec == "bf16" else torch.float16).float().cpu().numpy()
    best = A.argmin(2)
    i = np.clip(best, 1, max(1, D - 2))[..., None]
    take = lambda k: np.take_along_axis(A, np.clip(i + k, 0, D - 1), 2)[..., 0]  # noqa: E731
    a, b, c = take(-1), take(0), take(1)
    den = np.float32(2) * a + np.float32(2) * c - np.float32(4) * b
    ok = (best > 0) & (best < D - 1) & (den > 0)
    sub = best + np.where(ok, (a - c) / np.where(ok, den, np.float32(1)), np.float32(0)).astype(np.float32)
    assert np.array_equal(di.cpu().numpy(), best)
    np.testing.assert_allclose(ds.cpu().numpy(), sub, rtol=0, atol=2.0 ** -22 * max(1, D))


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("H,W,C,D", [(24, 40, 3, 49), (24, 40, 1, 128), (40, 200, 3, 256), (60, 300, 3, 241),
                                     (61, 310, 1, 256), (120, 300, 3, 256)])
def test_cost_groups_divided_over_ctas(fbs, prec, H, W, C, D):
    """Frames whose tiles leave SMs without a CTA share out the groups of 16 disparities (one round of the warps and
    more, one CTA with the rows after the costs only), larger ones do not."""
    test_radius_zero_maps_are_those_of_the_rounded_fp32_costs(fbs, prec, H, W, C, D)
