"""Storage conversion of array sources at the edges of its kernels' tiles: rows shorter and longer than a
block, ragged offset bricks, records whose channel count is and is not a multiple of the load width, sources
that start off a 16-byte boundary, host sources, and NaN / signed zeros / large values. Stored bytes, scales,
offsets, occupancy bits and brick distances are integers or exact binary32 results: bit-exact against the
oracle's quantiser and brick definitions."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fnr():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    torch.cuda.set_device(0)
    return fnr


def device_bytes(ptr, nbytes):
    import torch

    class _V:
        __cuda_array_interface__ = {"shape": (nbytes,), "typestr": "|u1", "data": (ptr, False), "version": 3}

    return torch.as_tensor(_V(), device="cuda").cpu().numpy()


def source(k, D, seed):
    """Densities mostly 0, some negative or NaN; channels over four decades with NaN, +-0 and a constant brick."""
    rng = np.random.default_rng(seed)
    n, nch = k ** 3, 3 * D
    sigma = np.where(rng.random(n) < 0.1, rng.uniform(-5, 50, n), 0).astype(np.float32)
    sigma[rng.random(n) < 0.01] = np.nan
    uvw = (rng.standard_normal((n, nch)) * 10.0 ** rng.uniform(-2, 2, nch)).astype(np.float32)
    uvw[rng.random((n, nch)) < 0.01] = 0.0
    uvw[rng.random((n, nch)) < 0.002] = -0.0
    uvw[rng.random((n, nch)) < 0.005] = np.nan
    if nch > 3:
        uvw[:, 1] = np.nan  # a channel with no value at all
        uvw[:, 2] = 0.75    # and a constant one
    beta = rng.standard_normal((5, 5, D)).astype(np.float32)
    return sigma, uvw.reshape(-1), beta


def brick_distance(occ, k, B, J):
    """Chebyshev distance in jump bricks of J cells, capped at 16, from the occupancy of bricks of B cells."""
    nb, nj, m = -(-k // B), -(-k // J), J // B
    pad = np.zeros((nj * m,) * 3, bool)
    pad[:nb, :nb, :nb] = occ.reshape(nb, nb, nb) != 0
    s = pad.reshape(nj, m, nj, m, nj, m).any(axis=(1, 3, 5))
    d = np.zeros((nj,) * 3, np.uint8)
    for _ in range(16):
        d += ~s
        for ax in range(3):
            g = np.pad(s, [(1, 1) if a == ax else (0, 0) for a in range(3)])
            s = sum(np.take(g, range(i, i + nj), axis=ax).astype(np.uint8) for i in range(3)) > 0
    return d.reshape(-1)


@pytest.mark.parametrize("k,D,brick", [(1, 1, 0), (5, 3, 1), (8, 8, 0), (24, 4, 2), (33, 2, 0), (37, 8, 16), (64, 6, 4),
                                       (65, 5, 0), (70, 16, 0), (96, 8, 1), (257, 1, 0)])
@pytest.mark.parametrize("where", ["device", "device+4", "host"])
def test_stored_bytes(fnr, k, D, brick, where):
    import torch
    sigma, uvw, beta = source(k, D, 100 * k + D)
    if where == "host":
        arrays = (sigma, uvw, beta)
    else:
        def put(a):  # "+4": the array starts one float past an aligned address
            off = where == "device+4"
            t = torch.zeros(a.size + 1, device="cuda")
            t[int(off):a.size + int(off)] = torch.from_numpy(a.reshape(-1)).cuda()
            return t[int(off):a.size + int(off)]
        arrays = tuple(put(a) for a in (sigma, uvw, beta))
    ctx = fnr.fnr_context_create(0, 0)
    try:
        for prec in (fnr.FNR_PREC_FP32, fnr.FNR_PREC_FP16, fnr.FNR_PREC_FP8_E4M3):
            cache = fnr.fnr_build_cache(ctx, fnr.make_desc(k, D, 5, prec, min(prec, 1), occupancy_brick=brick), *arrays)
            lay = fnr.fnr_cache_get_layout(cache)
            es = (4, 2, 1)[prec]
            want = oracle.quantize_cache(k, D, 5, sigma, uvw, beta, prec, min(prec, 1))
            as_bytes = lambda a: np.ascontiguousarray(a).view(np.uint8).reshape(-1)
            if prec == fnr.FNR_PREC_FP32:
                got = device_bytes(lay.sigma_dev, 4 * k ** 3).view(np.float32)
                assert np.array_equal(got, want.sigma)
            else:
                assert np.array_equal(device_bytes(lay.sigma_dev, es * k ** 3), as_bytes(want.sigma))
            rec = device_bytes(lay.uvw_dev, k ** 3 * lay.record_stride).reshape(k ** 3, lay.record_stride)
            assert np.all(rec[:, 3 * D * es:] == 0)
            ref = want.uvw.reshape(k ** 3, 3 * D)
            got = np.ascontiguousarray(rec[:, :3 * D * es]).view(ref.dtype)
            nan = np.isnan(uvw.reshape(k ** 3, 3 * D))
            assert np.array_equal(got[~nan], ref[~nan])
            value = {0: lambda a: a, 1: lambda a: a.view(np.float16)}.get(prec, lambda a: oracle.e4m3_decode(a))
            assert np.all(np.isnan(value(got[nan])))
            if prec == fnr.FNR_PREC_FP8_E4M3:
                nbo = -(-k // lay.offset_brick)
                offs = device_bytes(lay.offsets_dev, nbo ** 3 * lay.offset_stride * 2).view(np.uint16)
                offs = offs.reshape(nbo ** 3, lay.offset_stride)
                assert np.array_equal(offs[:, :3 * D].reshape(-1) & 0x7fff, want.offsets & 0x7fff)
                assert np.array_equal(offs[:, :3 * D].reshape(-1).view(np.float16), want.offsets.view(np.float16))
                assert np.all(offs[:, 3 * D:] == 0)
                assert np.array_equal(device_bytes(lay.scales_dev, 4 * (1 + 3 * D)), as_bytes(want.scales))
            B, J = lay.occupancy_brick, lay.distance_brick
            nb, nj = -(-k // B), -(-k // J)
            occ = oracle.brick_occupancy(k, B, oracle.positive_density(want))
            words = device_bytes(lay.occupancy_dev, -(-nb ** 3 // 32) * 4)
            bits = np.unpackbits(words, bitorder="little")
            assert np.array_equal(bits[:nb ** 3], occ) and not bits[nb ** 3:].any()
            assert np.array_equal(device_bytes(lay.brick_distance_dev, nj ** 3), brick_distance(occ, k, B, J))
            fnr.fnr_cache_free(ctx, cache)
    finally:
        fnr.fnr_context_destroy(ctx)
