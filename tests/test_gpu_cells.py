"""Renders that write every sample's (or walked) cell run kernels of their own. Their RGBA and counters equal those of
the same render without cells bit for bit, over sample counts around the group sizes, record lengths on both sides of
each change of group size and residency, ragged images and several views; the cells themselves are checked against
the oracle by the other tests."""

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("D", [1, 6, 7, 8, 9, 12, 13, 16])
def test_with_and_without_cells(prec, D):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    k, l = 14, 8
    rng = np.random.default_rng(100 * prec + D)
    sig = np.where(rng.random(k ** 3) < 0.5, rng.choice([0.4, 3.0], k ** 3), 0.0).astype(np.float32)
    sig.reshape(k, k, k)[: k // 2, :, : k // 2] = 0.0
    uvw = rng.standard_normal(k ** 3 * 3 * D).astype(np.float32)
    beta = rng.standard_normal(l * l * D).astype(np.float32)
    cams = [scenegen.cameras(D, 1, 37, 21)[0], scenegen.cameras(D + 1, 1, 8, 5, fov_deg=100.0)[0]]
    npix = 37 * 21 + 8 * 5
    ctx = fnr.fnr_context_create(0, 0)
    try:
        for layout in (fnr.FNR_LAYOUT_DENSE, fnr.FNR_LAYOUT_BRICKS):
            cache = fnr.fnr_build_cache(ctx, fnr.make_desc(k, D, l, prec, 0, occupancy_brick=4, layout=layout), sig, uvw,
                                        beta)
            calls = [(N, thr, skip, False) for N, thr in ((1, 0.0), (5, 0.0), (6, 1e-2), (8, 0.0), (9, 1e-2), (61, 1e-4))
                     for skip in (False, True)]
            if layout == fnr.FNR_LAYOUT_DENSE:
                calls += [(N, thr, skip, True) for N, thr in ((3, 0.0), (9, 1e-2), (3 * k, 0.0), (3 * k, 0.5))
                          for skip in (False, True)]
            for N, thr, skip, voxels in calls:
                p = fnr.make_params(N, t_thr=thr, skip_empty=skip, voxels=voxels)
                got = []
                for cells in (None, torch.full((npix * N,), -9, device="cuda", dtype=torch.int32)):
                    rgba = torch.full((npix * 4,), 7.0, device="cuda")
                    st = torch.full((npix * 4,), -5, device="cuda", dtype=torch.int32)
                    fnr.fnr_render(ctx, cache, cams, p, rgba, st, cells)
                    got.append((rgba, st))
                torch.cuda.synchronize()
                case = (layout, N, thr, skip, voxels)
                assert torch.equal(got[0][0], got[1][0]), case
                assert torch.equal(got[0][1], got[1][1]), case
                assert not bool((cells == -9).any()), case
            fnr.fnr_cache_free(ctx, cache)
    finally:
        fnr.fnr_context_destroy(ctx)
