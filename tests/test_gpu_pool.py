"""Temporaries from a context's pool: builds and uncached renders issued at once from several threads on their own
streams (which share the pool's memory) give the bytes that the same calls give one after the other."""

import threading

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_threads", [2, 4])
def test_concurrent_builds_share_the_pool(n_threads):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr

    def device_bytes(ptr, n):
        class _V:
            __cuda_array_interface__ = {"shape": (n,), "typestr": "|u1", "data": (ptr, False), "version": 3}
        return torch.as_tensor(_V(), device="cuda").cpu().numpy()

    dev = lambda layers: [(torch.from_numpy(W.view(np.int16)).cuda(), torch.from_numpy(b).cuda()) for W, b in layers]
    pos, dirn = dev(scenegen.mlp_weights(3, scenegen.FPOS_DIMS_D8, 0.05)), dev(scenegen.mlp_weights(4, scenegen.FDIR_DIMS_D8, 0.05))
    k, D, l = 40, 8, 12
    rng = np.random.default_rng(n_threads)
    work = []
    for i in range(n_threads):
        sig = torch.from_numpy(np.where(rng.random(k ** 3) < 0.1, 50.0, 0.0).astype(np.float32)).cuda()
        uvw = torch.from_numpy(rng.standard_normal(k ** 3 * 3 * D).astype(np.float32)).cuda()
        beta = torch.from_numpy(rng.standard_normal(l * l * D).astype(np.float32)).cuda()
        work.append((sig, uvw, beta, scenegen.cameras(i, 1, 30 + i, 20)[0]))
    torch.cuda.synchronize()
    ctx = fnr.fnr_context_create(0, 0)

    def calls(i, out):
        torch.cuda.set_device(0)
        stream = torch.cuda.Stream()
        sig, uvw, beta, cam = work[i]
        for rep in range(4):
            got = []
            for prec, layout in ((2, 0), (1, 1)):
                c = fnr.fnr_build_cache(ctx, fnr.make_desc(k, D, l, prec, 1, layout=layout), sig, uvw, beta, stream=stream)
                lay = fnr.fnr_cache_get_layout(c)
                cells = k ** 3 if layout == 0 else lay.n_bricks * lay.occupancy_brick ** 3
                with torch.cuda.stream(stream):
                    got.append(device_bytes(lay.uvw_dev, cells * lay.record_stride).copy())
                fnr.fnr_cache_free(ctx, c)
            c = fnr.fnr_build_cache_mlp(ctx, fnr.make_desc(20, D, l), pos, dirn, stream=stream)
            lay = fnr.fnr_cache_get_layout(c)
            with torch.cuda.stream(stream):
                got.append(device_bytes(lay.uvw_dev, 20 ** 3 * lay.record_stride).copy())
            fnr.fnr_cache_free(ctx, c)
            with torch.cuda.stream(stream):
                rgba = torch.zeros(cam["W"] * cam["H"] * 4, device="cuda")
                fnr.fnr_render_mlp(ctx, pos, dirn, D, cam, fnr.make_params(24), rgba, stream=stream)
                got.append(rgba.cpu().numpy())
            out.append(got)

    try:
        serial = [[] for _ in range(n_threads)]
        for i in range(n_threads):
            calls(i, serial[i])
        together = [[] for _ in range(n_threads)]
        threads = [threading.Thread(target=calls, args=(i, together[i])) for i in range(n_threads)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for a, b in zip(serial, together):
            assert len(a) == len(b) == 4
            for x, y in zip(a, b):
                for p, q in zip(x, y):
                    assert np.array_equal(p, q)
        assert fnr.fnr_context_used_bytes(ctx) == 0
    finally:
        fnr.fnr_context_destroy(ctx)
