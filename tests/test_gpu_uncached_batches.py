"""The uncached render's batches of rays (8 Mi samples each, or 16 Ki rays if that is more).

A view of several batches equals, byte for byte, the same rays rendered as strips of one batch each: shifting the
principal point by whole rows leaves (py + 1/2) - cy, and so every ray, the same binary32 number, and neither the
networks' products nor the compositing of a ray depend on the rays around it. A render that fails on the device
leaves the caller's arrays as they were, whatever the number of batches."""

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

N = 512  # 16 Ki rays are 8 Mi samples
ONE, SEVERAL = (211, 38), (211, 190)  # 8,018 and 40,090 rays: one batch, and three of which the last is ragged


@pytest.fixture(scope="module")
def fnr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    torch.cuda.set_device(0)
    return fnr


def networks(D):
    import torch
    out = []
    for seed, dims in ((D, [60, 32, 1 + 3 * D]), (D + 50, [24, 16, D])):
        layers = scenegen.mlp_weights(seed, dims, bias_scale=0.3)
        layers[-1][1][0] += 2.0  # densities at which some rays end early
        out.append([(torch.from_numpy(W.view(np.int16)).cuda(), torch.from_numpy(b).cuda()) for W, b in layers])
    return out


def arrays(W, H):
    import torch
    return (torch.full((W * H * 4,), 7.0, device="cuda"), torch.full((W * H * 4,), -5, device="cuda", dtype=torch.int32))


def camera(size, row=0):
    cam = scenegen.cameras(3, 1, *SEVERAL)[0]
    return dict(cam, W=size[0], H=size[1], cy=np.float32(cam["cy"] - row))


@pytest.mark.parametrize("with_stats", [True, False])
@pytest.mark.parametrize("D,n", [(1, N), (8, N), (4, N + 190)])
def test_batches_equal_strips(fnr, D, n, with_stats):
    import torch
    nets, p = networks(D), fnr.make_params(n, t_thr=0.3)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        def render(cam):
            rgba, stats = arrays(cam["W"], cam["H"])
            fnr.fnr_render_mlp(ctx, *nets, D, cam, p, rgba, stats if with_stats else None)
            return rgba, stats

        whole = render(camera(SEVERAL))
        strips = [render(camera(ONE, row)) for row in range(0, SEVERAL[1], ONE[1])]
        torch.cuda.synchronize()
        for got, want in zip(whole, zip(*strips)):
            assert torch.equal(got, torch.cat(want))
        seen = torch.cat([s for _, s in strips]).reshape(-1, 4)
        if with_stats:
            assert bool((seen[:, 0] < n).any()) and bool((seen[:, 3] == -1).all())
        else:
            assert bool((seen == -5).all())
        assert fnr.fnr_context_used_bytes(ctx) == 0
    finally:
        fnr.fnr_context_destroy(ctx)


@pytest.mark.parametrize("size", [ONE, SEVERAL])
def test_failed_render_leaves_the_arrays(fnr, size):
    import torch
    nets, p, cam = networks(8), fnr.make_params(N), camera(size)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        rgba, stats = arrays(*size)
        fnr.fnr_testing_mlp_fault(1 << 12, 0)  # F_pos never gets its first weights
        with pytest.raises(fnr.FnrError) as ei:
            fnr.fnr_render_mlp(ctx, *nets, 8, cam, p, rgba, stats)
        assert ei.value.status == fnr.FNR_ERR_DEVICE and "ran out" in str(ei.value)
        torch.cuda.synchronize()
        assert bool((rgba == 7.0).all()) and bool((stats == -5).all())
        fnr.fnr_render_mlp(ctx, *nets, 8, cam, p, rgba, stats)
        torch.cuda.synchronize()
        assert not bool((rgba.reshape(-1, 4) == 7.0).any()) and not bool((stats == -5).any())
    finally:
        fnr.fnr_context_destroy(ctx)


def test_budget_is_charged_for_one_batch(fnr):
    """The samples of the view would take 2.3 GB at once, a batch's 0.8: a budget between the two admits the view, one
    below the batch does not, and either way nothing stays charged."""
    import torch
    nets, p, cam = networks(8), fnr.make_params(N), camera(SEVERAL)
    images = []
    for budget in (0, 1 << 30):
        ctx = fnr.fnr_context_create(0, budget)
        rgba, stats = arrays(*SEVERAL)
        fnr.fnr_render_mlp(ctx, *nets, 8, cam, p, rgba, stats)
        torch.cuda.synchronize()
        images.append(rgba)
        assert fnr.fnr_context_used_bytes(ctx) == 0
        fnr.fnr_context_destroy(ctx)
    assert torch.equal(*images)
    ctx = fnr.fnr_context_create(0, 1 << 29)
    with pytest.raises(fnr.FnrError) as ei:
        fnr.fnr_render_mlp(ctx, *nets, 8, cam, p, rgba, stats)
    assert ei.value.status == fnr.FNR_ERR_BUDGET and fnr.fnr_context_used_bytes(ctx) == 0
    fnr.fnr_context_destroy(ctx)


@pytest.mark.parametrize("size", [ONE, SEVERAL])
def test_view_past_the_box(fnr, size):
    """No ray reaches the box: F_pos has no samples at all, and the image is the background."""
    import torch
    nets, cam = networks(8), camera(size)
    cam["c2w"] = np.array(cam["c2w"], np.float32)
    cam["c2w"][3::4] += 100.0
    p = fnr.make_params(N, bg=(0.25, 0.5, 0.75))
    ctx = fnr.fnr_context_create(0, 0)
    try:
        rgba, stats = arrays(*size)
        fnr.fnr_render_mlp(ctx, *nets, 8, cam, p, rgba, stats)
        want = torch.tensor([0.25, 0.5, 0.75, 0.0], device="cuda")
        assert bool((rgba.reshape(-1, 4) == want).all())
        assert bool((stats.reshape(-1, 4) == torch.tensor([N, 0, 0, -1], device="cuda", dtype=torch.int32)).all())
    finally:
        fnr.fnr_context_destroy(ctx)
