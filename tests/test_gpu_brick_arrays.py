"""Sparse caches built from device arrays, whose records are converted straight into the brick pools, against the dense
cache of the same arrays: pools gathered through the page table byte for byte (cells past the grid's edge and record
padding 0), and the direction cache, scales, offsets, occupancy bits and brick distances. Load widths of 1, 2 and 4
floats (by record length and by sources off a 16-byte boundary), ragged edge bricks, and a cache without a brick.
The dense stored bytes are checked against the oracle by the conversion tests."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fnr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    torch.cuda.set_device(0)
    return fnr


def device_bytes(ptr, nbytes):
    import torch
    if nbytes == 0:
        return np.zeros(0, np.uint8)

    class _V:
        __cuda_array_interface__ = {"shape": (nbytes,), "typestr": "|u1", "data": (ptr, False), "version": 3}

    return torch.as_tensor(_V(), device="cuda").cpu().numpy()


@pytest.mark.parametrize("k,brick", [(9, 4), (33, 0), (40, 8), (65, 0)])
@pytest.mark.parametrize("D", [1, 2, 3, 8, 16])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_pools_equal_the_dense_cache(fnr, k, brick, D, shift):
    import torch
    rng = np.random.default_rng(1000 * k + 10 * D + shift)
    l, nch = 5, 3 * D
    sigma = np.where(rng.random(k ** 3) < 0.002, rng.uniform(0, 50, k ** 3), 0).astype(np.float32)
    sigma[0], sigma[-1] = 1.0, 2.0  # the first cell and the last, in the ragged corner brick
    uvw = (rng.standard_normal((k ** 3, nch)) * 10.0 ** rng.uniform(-2, 2, nch)).astype(np.float32)
    beta = rng.standard_normal(l * l * D).astype(np.float32)

    def put(a):  # starts `shift` floats past an aligned address
        t = torch.zeros(a.size + 4, device="cuda")
        t[shift:a.size + shift] = torch.from_numpy(a.reshape(-1)).cuda()
        return t[shift:a.size + shift]

    ctx = fnr.fnr_context_create(0, 0)
    try:
        for empty in (False, True):
            arrays = tuple(put(a) for a in (sigma * np.float32(not empty), uvw, beta))
            for prec in (fnr.FNR_PREC_FP32, fnr.FNR_PREC_FP16, fnr.FNR_PREC_FP8_E4M3):
                es = (4, 2, 1)[prec]
                desc = lambda layout: fnr.make_desc(k, D, l, prec, min(prec, 1), occupancy_brick=brick, layout=layout)
                dense = fnr.fnr_build_cache(ctx, desc(fnr.FNR_LAYOUT_DENSE), *arrays)
                pools = fnr.fnr_build_cache(ctx, desc(fnr.FNR_LAYOUT_BRICKS), *arrays)
                a, b = fnr.fnr_cache_get_layout(dense), fnr.fnr_cache_get_layout(pools)
                B = a.occupancy_brick
                nb, nj = -(-k // B), -(-k // a.distance_brick)
                same = [("beta_dev", l * l * D * (4 if prec == 0 else 2)), ("cos_theta_dev", 4 * l), ("phi_key_dev", 4 * l),
                        ("occupancy_dev", -(-nb ** 3 // 32) * 4), ("brick_distance_dev", nj ** 3)]
                if prec == fnr.FNR_PREC_FP8_E4M3:
                    nbo = -(-k // a.offset_brick)
                    same += [("scales_dev", 4 * (1 + nch)), ("offsets_dev", nbo ** 3 * a.offset_stride * 2)]
                for name, n in same:
                    assert np.array_equal(device_bytes(getattr(a, name), n), device_bytes(getattr(b, name), n)), name
                words = device_bytes(a.occupancy_dev, -(-nb ** 3 // 32) * 4)
                occ = np.unpackbits(words, bitorder="little")[:nb ** 3] != 0
                assert b.n_bricks == occ.sum() and (b.n_bricks == 0) == empty
                page = device_bytes(b.page_table_dev, 4 * nb ** 3).view(np.int32)
                assert np.array_equal(page, np.where(occ, np.cumsum(occ) - 1, -1))
                # dense planes, padded with zeros to whole bricks, in pool order
                for da, db, width in ((a.sigma_dev, b.sigma_dev, es), (a.uvw_dev, b.uvw_dev, a.record_stride)):
                    plane = np.zeros((nb * B,) * 3 + (width,), np.uint8)
                    plane[:k, :k, :k] = device_bytes(da, k ** 3 * width).reshape(k, k, k, width)
                    bricks = plane.reshape(nb, B, nb, B, nb, B, width).transpose(0, 2, 4, 1, 3, 5, 6)
                    want = bricks.reshape(nb ** 3, -1)[occ].reshape(-1)
                    assert np.array_equal(device_bytes(db, want.size), want)
                for c in (dense, pools):
                    fnr.fnr_cache_free(ctx, c)
    finally:
        fnr.fnr_context_destroy(ctx)
