"""The voxel walk's divisions by the ray direction, at the edges of the range in which they go through reciprocals.

The walk divides by u_a = d_a k / (bmax_a - bmin_a) through 1 / u_a while 2^-60 <= |u_a| <= 2^60 and the eye's grid
coordinate is 0 or in the same range, and with the general division otherwise, warp by warp. Boxes here put the rays
inside that range, at its two ends and outside it, with eyes on a face of the box (coordinate 0), next to one, and
rays along the axes. Bar: that of the walk's other tests -- walked cells and counters equal to the oracle's, RGBA
within 1e-5.
"""

import numpy as np
import pytest

import oracle
import scenegen
from test_gpu_voxels import TOL, check, ctx, fnr, oparams, render  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu

K, D, L = 16, 2, 6


def scene_arrays(size):
    """Cells of density 0 (most), low and high, in units in which a cell of the box is `size` long."""
    rng = np.random.Generator(np.random.PCG64(5))
    sig = np.where(rng.random(K ** 3) < 0.7, 0.0, rng.choice([0.05, 0.5, 3.0], K ** 3)) / size
    uvw = rng.uniform(-2.0, 2.0, (K ** 3, 3 * D))
    beta = rng.uniform(-1.0, 1.0, (L * L, D))
    return sig.astype(np.float32), uvw.astype(np.float32), beta.astype(np.float32)


@pytest.mark.parametrize("edge", [3.0, 2.0 ** -56, 2.0 ** -57, 2.0 ** -61, 2.0 ** 62, 2.0 ** 64, 2.0 ** 66])
@pytest.mark.parametrize("skip", [False, True])
def test_walk_division_range(fnr, ctx, edge, skip):  # noqa: F811
    h = edge / 2
    sig, uvw, beta = scene_arrays(edge / K)
    box = dict(bmin=(-h, -h, -h), bmax=(h, h, h))
    cache = fnr.fnr_build_cache(ctx, fnr.make_desc(K, D, L, occupancy_brick=4, **box), sig, uvw.reshape(-1),
                                beta.reshape(-1))
    try:
        oc = oracle.Cache(K, D, L, sig, uvw, beta, **box).set_occupancy(4)
        eyes = [(1.9, 1.2, 1.4),                  # every axis sloped
                (-1.0, 0.3, 0.2),                 # on a face: coordinate 0
                (-1.0 + 2.0 ** -20, -1.0, -1.0),  # next to a corner
                (0.1, 0.2, 0.3)]                  # inside
        for eye in eyes:
            cam = scenegen.look_at_camera(eye, 13, 9)
            pose = cam["c2w"].reshape(3, 4).astype(np.float64)
            pose[:, 3] = np.array(eye) * h
            along = np.hstack([np.eye(3), [[0.1 * h], [0.2 * h], [1.5 * h]]])  # its middle column and row: u_a = 0
            for c2w in (pose, along):
                cam["c2w"] = c2w.astype(np.float32).reshape(12)
                p = fnr.make_params(3 * K, t_near=0.0, t_far=4.0 * edge, t_thr=1e-3, voxels=True, skip_empty=skip)
                got = render(fnr, ctx, cache, cam, p)
                ref = oracle.render_image(oc, cam, oparams(p), want_cells=True)
                check(got, ref, TOL)
                jump = render(fnr, ctx, cache, cam, p, with_cells=False)
                assert np.array_equal(jump[0], got[0]) and np.array_equal(jump[1], got[1])
    finally:
        fnr.fnr_cache_free(ctx, cache)
