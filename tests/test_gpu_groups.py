"""The march's sample groups (5 or 6 by precision and record length) at their edges: rays with fewer samples than a
group, exactly one, one more, and a last group cut off by the far end or by termination; record lengths on both sides
of each change of group size and residency. Cells, counters and the direction cell equal the oracle's; RGBA within
1e-5, as for the other renders."""

import numpy as np
import pytest

import oracle
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("D", [4, 6, 7, 8, 9, 12, 13])
def test_group_edges(prec, D):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    k, l, W, H = 14, 8, 37, 21
    rng = np.random.default_rng(100 * prec + D)
    sig = np.where(rng.random(k ** 3) < 0.5, rng.choice([0.4, 3.0], k ** 3), 0.0).astype(np.float32)
    sig.reshape(k, k, k)[: k // 2, :, : k // 2] = 0.0
    uvw = rng.standard_normal((k ** 3, 3 * D)).astype(np.float32)
    beta = rng.standard_normal((l, l, D)).astype(np.float32)
    cam = scenegen.cameras(D, 1, W, H)[0]
    ctx = fnr.fnr_context_create(0, 0)
    try:
        oc = oracle.quantize_cache(k, D, l, sig, uvw, beta, prec, 0).set_occupancy(4)
        for layout in (fnr.FNR_LAYOUT_DENSE, fnr.FNR_LAYOUT_BRICKS):
            cache = fnr.fnr_build_cache(ctx, fnr.make_desc(k, D, l, prec, 0, occupancy_brick=4, layout=layout), sig,
                                        uvw.reshape(-1), beta.reshape(-1))
            for N, thr in ((1, 0.0), (4, 0.0), (5, 0.0), (6, 0.0), (7, 1e-2), (11, 1e-2), (40, 1e-2), (61, 1e-4)):
                for skip in ((False, True) if layout == fnr.FNR_LAYOUT_DENSE else (True,)):
                    rgba = torch.zeros(W * H * 4, device="cuda")
                    st = torch.zeros(W * H * 4, device="cuda", dtype=torch.int32)
                    cells = torch.zeros(W * H * N, device="cuda", dtype=torch.int32)
                    p = fnr.make_params(N, t_thr=thr, skip_empty=skip)
                    fnr.fnr_render(ctx, cache, [cam], p, rgba, st, cells)
                    torch.cuda.synchronize()
                    ref, rst, rcells = oracle.render_image(
                        oc, cam, oracle.params_struct(N, t_thr=thr, skip_empty=skip), want_cells=True)
                    assert np.array_equal(cells.cpu().numpy().reshape(H, W, N), rcells)
                    assert np.array_equal(st.cpu().numpy().reshape(H, W, 4), rst)
                    assert np.max(np.abs(rgba.cpu().numpy().reshape(H, W, 4) - ref)) <= 1e-5
    finally:
        fnr.fnr_context_destroy(ctx)
