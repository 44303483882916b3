"""Failure detection without a device fault: a bounded wait that runs out, an
injected launch failure and a corrupt autotune cache, each reported through
the C ABI, with the context usable afterwards."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fbs():
    from paper_1807_02044_gb300 import build as b
    b.build()
    import paper_1807_02044_gb300 as m
    return m


def _pair(seed=1, H=96, W=160):
    rng = np.random.default_rng(seed)
    L = rng.integers(0, 256, size=(H, W, 3)).astype(np.uint8)
    R = np.roll(L, -6, axis=1)
    return torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()


def _run(fbs, ctx, dl, dr):
    di, ds = ctx.compute_disparity(dl, dr, 64, 7, 7.0, 12.0)
    torch.cuda.synchronize()
    return di, ds


@pytest.mark.parametrize("prec", ["bf16", "f16"])
def test_wait_limit_runs_out_and_the_context_recovers(fbs, prec):
    """A limit of about 100 ns is shorter than any pipeline hand-off of the
    tensor-core aggregation, so its waits run out: the kernel stops, drains
    what it issued and frees its tensor memory, and fbs_sync reports
    FBS_ERR_TIMEOUT.  With the default limit restored the same context gives
    the results of a fresh one."""
    p = fbs.FBS_PREC_BF16 if prec == "bf16" else fbs.FBS_PREC_F16
    dl, dr = _pair()
    with fbs.Context(0, prec=p) as ref:
        di0, ds0 = _run(fbs, ref, dl, dr)
        fbs.fbs_sync(ref.ctx)
    with fbs.Context(0, prec=p) as ctx:
        fbs.fbs_set_wait_limit(ctx.ctx, 1e-7)
        _run(fbs, ctx, dl, dr)
        with pytest.raises(fbs.FBSError) as ei:
            fbs.fbs_sync(ctx.ctx)
        assert ei.value.status == fbs.FBS_ERR_TIMEOUT
        assert "bounded wait" in fbs.fbs_last_error(ctx.ctx)
        fbs.fbs_set_wait_limit(ctx.ctx, 0.0)
        di, ds = _run(fbs, ctx, dl, dr)
        fbs.fbs_sync(ctx.ctx)
        assert torch.equal(di, di0) and torch.equal(ds, ds0)
        with pytest.raises(fbs.FBSError):
            fbs.fbs_set_wait_limit(ctx.ctx, -1.0)


def test_convolution_wait_runs_out_and_stores_nothing(fbs):
    """A limit of a clock cycle is over before the MMAs of a tile can have
    completed.  Whatever a warp whose wait ran out leaves unstored still holds
    the value of the first call on the same pair, so the activations and the
    outputs stay bit for bit what they were, while fbs_sync reports
    FBS_ERR_TIMEOUT; with the default limit the context computes again."""
    H, W, D = 96, 160, 64
    (dl, dr), (el, er) = _pair(3), _pair(4)
    P = (H // 4) * (W // 4)
    with fbs.Context(0) as ctx:
        fbs.fbs_band_net_load(ctx.ctx, fbs.default_band_net_path())

        def forward(left, right, out):
            fbs.fbs_band_net_forward(ctx.ctx, left, right, H, W, 3, D, *out)
            torch.cuda.synchronize()
            return [o.clone() for o in out]

        def outputs():
            out = [torch.full(s, -7.0, device="cuda") for s in ((H // 4, W // 4, 2), (H, W), (H, W))]
            torch.cuda.synchronize()   # the call runs on the context's own stream
            return out

        def trace():
            acts = torch.empty(P * (8 + 5 * 32 + 2), device="cuda")
            torch.cuda.synchronize()
            fbs.fbs_band_net_trace(ctx.ctx, acts, None)
            torch.cuda.synchronize()
            return acts

        out, other = outputs(), outputs()
        first, other_first = forward(dl, dr, out), forward(el, er, other)
        assert all(torch.equal(a, b) for a, b in zip(first, forward(dl, dr, out)))
        acts = trace()
        fbs.fbs_sync(ctx.ctx)
        fbs.fbs_set_wait_limit(ctx.ctx, 1e-9)
        late = forward(dl, dr, out)
        with pytest.raises(fbs.FBSError) as ei:
            fbs.fbs_sync(ctx.ctx)
        assert ei.value.status == fbs.FBS_ERR_TIMEOUT and "code 21" in fbs.fbs_last_error(ctx.ctx)
        assert torch.equal(trace(), acts)
        assert all(torch.equal(a, b) for a, b in zip(first, late))
        fbs.fbs_set_wait_limit(ctx.ctx, 0.0)
        assert all(torch.equal(a, b) for a, b in zip(other_first, forward(el, er, outputs())))
        fbs.fbs_sync(ctx.ctx)


@pytest.mark.parametrize("form", ["path", "lr", "unaligned", "batch0", "batch3", "batch4", "band"])
def test_fp32_aggregation_wait_runs_out_and_stores_nothing(fbs, form):
    """A limit of a clock cycle is over before a copied cost row can have landed:
    the CTAs of an SM ask for 128 KB of rows at once, and with radius 0 they have
    a few hundred cycles of work before they wait for them; the 4-byte copies
    take longer to issue, and there (radius 1) the first warps that are done with
    a slot wait for the others before they refill it.
    A tile whose wait ran out lets its copies land and stores nothing, so it
    still holds the maps of the first call on the same inputs, and every other
    tile computes them again: the outputs stay bit for bit what they were,
    while fbs_sync reports FBS_ERR_TIMEOUT; with the default limit the context
    computes other inputs like a fresh one.  Forms: TMA rows, both views, 4-byte
    copies (D = 255), the persistent (0, 3) and a branched (4) batch plan, bands."""
    H, W, D, r = 240, 640, 256, int(form == "unaligned")
    (dl, dr), (el, er) = _pair(3, H, W), _pair(4, H, W)
    cost = torch.rand((2, H, W, 255), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    centre, conf = torch.full((H, W), 6.0, device="cuda"), (torch.arange(W, device="cuda") < W // 2).float().repeat(H, 1)
    torch.cuda.synchronize()

    def outputs():
        return [torch.full((H, W), -7, dtype=t, device="cuda") for t in (torch.int32, torch.float32) * 2]

    def call(ctx, left, right, out):
        st = torch.cuda.current_stream()
        pair = dict(left=left, right=right, H=H, W=W, C=3, D=D, radius=r, sigma_s=2.0, sigma_r=12.0, tau=0.0,
                    disp_int=out[0], disp_subpix=out[1])
        if form == "path":
            fbs.fbs_compute_disparity(ctx.ctx, left, right, H, W, 3, D, r, 2.0, 12.0, 0.0, out[0], out[1], st)
        elif form == "lr":
            fbs.fbs_compute_disparity_lr(ctx.ctx, left, right, H, W, 3, D, r, 2.0, 12.0, 0.0, *out, False, st)
        elif form == "unaligned":
            c = cost[0 if left is dl else 1]
            fbs.fbs_aggregate(ctx.ctx, c, left, H, W, 3, 255, r, 2.0, 12.0, None, out[0], out[1], st)
        elif form == "band":
            fbs.fbs_compute_disparity_banded(ctx.ctx, pair, centre, conf, 3, 0.5, st)
        else:
            pairs = [pair, dict(pair, radius=1, disp_int=out[2], disp_subpix=out[3])]
            fbs.fbs_batch_set_plan(ctx.ctx, pairs, int(form[5:]))
            fbs.fbs_compute_disparity_batched(ctx.ctx, pairs, st)
        torch.cuda.synchronize()
        return [o.clone() for o in out]

    with fbs.Context(0) as ref:
        want = call(ref, el, er, outputs())
        fbs.fbs_sync(ref.ctx)
    with fbs.Context(0) as ctx:
        out = outputs()
        first = call(ctx, dl, dr, out)
        fbs.fbs_sync(ctx.ctx)
        fbs.fbs_set_wait_limit(ctx.ctx, 1e-9)
        late = call(ctx, dl, dr, out)
        with pytest.raises(fbs.FBSError) as ei:
            fbs.fbs_sync(ctx.ctx)
        assert ei.value.status == fbs.FBS_ERR_TIMEOUT and "code 31" in fbs.fbs_last_error(ctx.ctx)
        assert all(torch.equal(a, b) for a, b in zip(first, late))
        fbs.fbs_set_wait_limit(ctx.ctx, 0.0)
        assert all(torch.equal(a, b) for a, b in zip(want, call(ctx, el, er, outputs())))
        fbs.fbs_sync(ctx.ctx)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_injected_launch_failure_is_reported_and_clears(fbs, prec):
    """An injected launch error surfaces as FBS_ERR_CUDA (an allocation error
    as FBS_ERR_OOM) with the error's text, launches nothing, and the next step
    runs normally."""
    p = fbs.FBS_PREC_F32 if prec == "f32" else fbs.FBS_PREC_BF16
    dl, dr = _pair(2)
    with fbs.Context(0, prec=p) as ctx:
        di0, ds0 = _run(fbs, ctx, dl, dr)
        fbs.fbs_sync(ctx.ctx)
        for err, status in ((700, fbs.FBS_ERR_CUDA), (2, fbs.FBS_ERR_OOM)):   # illegal address, memory allocation
            fbs.fbs_debug_fail_launches(ctx.ctx, err, 1)
            fbs.fbs_profile(ctx.ctx, 1)
            with pytest.raises(fbs.FBSError) as ei:
                _run(fbs, ctx, dl, dr)
            assert ei.value.status == status
            assert "injected" in fbs.fbs_last_error(ctx.ctx)
            launched = sum(fbs.fbs_profile_read(ctx.ctx, k)[1] for k in range(fbs.FBS_KERNEL_KINDS))
            fbs.fbs_profile(ctx.ctx, 0)
            assert launched == 0
            di, ds = _run(fbs, ctx, dl, dr)
            fbs.fbs_sync(ctx.ctx)
            assert torch.equal(di, di0) and torch.equal(ds, ds0)
        with pytest.raises(fbs.FBSError):
            fbs.fbs_debug_fail_launches(ctx.ctx, 0, 1)


def test_corrupt_autotune_cache_is_ignored(fbs, tmp_path):
    """Garbage, out-of-range plans and truncated lines in the autotune cache
    file are skipped: the batch still runs (autotuned afresh), gives the
    per-pair results, and a valid entry is appended."""
    from synth import random_batch_specs
    path = tmp_path / "tune.txt"
    path.write_bytes(b"\x00\xff garbage line\nt64x2 99\nf1 -3\nnot_a_number x\nt12")
    specs = random_batch_specs(11, n=3, wrange=(64, 128), hrange=(48, 96), dchoices=(16, 32), rchoices=(2, 4))
    pairs, ref = [], []
    with fbs.Context(0, prec=fbs.FBS_PREC_BF16, autotune_cache_path=str(path)) as ctx:
        for sp in specs:
            rng = np.random.default_rng(sp["seed"])
            L = rng.integers(0, 256, size=(sp["H"], sp["W"], 3)).astype(np.uint8)
            R = np.roll(L, -3, axis=1)
            dl, dr = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
            q = dict(left=dl, right=dr, H=sp["H"], W=sp["W"], C=3, D=sp["D"], radius=sp["radius"],
                     sigma_s=sp["sigma_s"], sigma_r=12.0, tau=30.0,
                     disp_int=torch.empty((sp["H"], sp["W"]), dtype=torch.int32, device="cuda"),
                     disp_subpix=torch.empty((sp["H"], sp["W"]), dtype=torch.float32, device="cuda"))
            pairs.append(q)
            di, ds = ctx.compute_disparity(dl, dr, sp["D"], sp["radius"], sp["sigma_s"], 12.0, 30.0)
            ref.append((di, ds))
        assert fbs.fbs_batch_plan(ctx.ctx, pairs) == -1
        fbs.fbs_compute_disparity_batched(ctx.ctx, pairs, torch.cuda.current_stream())
        torch.cuda.synchronize()
        fbs.fbs_sync(ctx.ctx)
        plan = fbs.fbs_batch_plan(ctx.ctx, pairs)
        assert plan >= 0
        for q, (di, ds) in zip(pairs, ref):
            assert torch.equal(q["disp_int"], di) and torch.equal(q["disp_subpix"], ds)
    last = path.read_bytes().splitlines()[-1].split()
    assert len(last) == 2 and int(last[1]) == plan
