"""The exact termination sum over densities at the edges of its fixed-point form: denormal, below 2^-32 (adds
nothing), with fractions at the last bit, integers past the significand's fraction, at and above 2^31 (saturated),
and the largest binary32. Every ray counter is bit-exact against the oracle, for uniform samples and for the voxel
walk (whose terms are binary32 products of density and length)."""

import numpy as np
import pytest

import oracle
import scenegen

pytestmark = pytest.mark.gpu

EDGES = np.array([1e-45, 1e-39, 2.0 ** -33, 2.0 ** -32, 3e-10, 0.2999999, 1.0, 1.5, 50.25, 8388608.5, 16777217.0, 2.0 ** 31 - 128,
                  2.0 ** 31, 3e9, 3.4e38], np.float32)


@pytest.mark.parametrize("t_thr", [1e-4, 0.5, 1e-30, 0.0])
@pytest.mark.parametrize("top", [4, 9, 12, 15])
def test_counters_over_density_edges(t_thr, top):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    k, D, l, W, H = 12, 2, 8, 40, 28
    rng = np.random.default_rng(top)
    sig = np.where(rng.random(k ** 3) < 0.6, EDGES[rng.integers(0, top, k ** 3)], 0).astype(np.float32)
    uvw = rng.standard_normal((k ** 3, 3 * D)).astype(np.float32)
    beta = rng.standard_normal((l, l, D)).astype(np.float32)
    cam = scenegen.cameras(top, 1, W, H)[0]
    ctx = fnr.fnr_context_create(0, 0)
    try:
        cache = fnr.fnr_build_cache(ctx, fnr.make_desc(k, D, l), sig, uvw.reshape(-1), beta.reshape(-1))
        oc = oracle.Cache(k, D, l, sig, uvw, beta)
        for voxels in (False, True):
            N = 3 * k if voxels else 70
            rgba = torch.zeros(W * H * 4, device="cuda")
            st = torch.zeros(W * H * 4, device="cuda", dtype=torch.int32)
            fnr.fnr_render(ctx, cache, [cam], fnr.make_params(N, t_thr=t_thr, voxels=voxels), rgba, st)
            torch.cuda.synchronize()
            ref, rst, _ = oracle.render_image(oc, cam, oracle.params_struct(N, t_thr=t_thr, voxels=voxels))
            assert np.array_equal(st.cpu().numpy().reshape(H, W, 4), rst)
            assert np.max(np.abs(rgba.cpu().numpy().reshape(H, W, 4) - ref)) <= 1e-5
    finally:
        fnr.fnr_context_destroy(ctx)
