"""Calls from a thread whose current CUDA context is another one on the same device (made through the driver API):
every entry point that launches or allocates makes the device's primary context current first, in which the caches
and the caller's buffers live, and gives the results that it gives elsewhere."""

import ctypes
import threading

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


def check(status):
    assert status == 0, f"driver call failed: {status}"


@pytest.fixture(scope="module")
def scene():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    torch.cuda.set_device(0)
    k, D, l = 20, 8, 6
    rng = np.random.default_rng(1)
    dev = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()
    arrays = (dev(np.where(rng.random(k ** 3) < 0.2, 3.0, 0.0)), dev(rng.standard_normal(k ** 3 * 3 * D)),
              dev(rng.standard_normal(l * l * D)))
    nets = [[(torch.from_numpy(W.view(np.int16)).cuda(), torch.from_numpy(b).cuda())
             for W, b in scenegen.mlp_weights(s, dims, 0.05)]
            for s, dims in ((3, [60, 32, 25]), (4, [24, 16, 8]))]
    ctx = fnr.fnr_context_create(0, 0)
    yield fnr, ctx, fnr.make_desc(k, D, l), arrays, nets, scenegen.cameras(2, 1, 40, 24)[0]
    fnr.fnr_context_destroy(ctx)


@pytest.mark.parametrize("call", ["render", "build", "build_mlp", "render_mlp", "load"])
def test_call_under_another_context(scene, call, tmp_path):
    import torch
    fnr, ctx, desc, arrays, nets, cam = scene
    p = fnr.make_params(48)
    rgba = torch.zeros(cam["W"] * cam["H"] * 4, device="cuda")
    cache = fnr.fnr_build_cache(ctx, desc, *arrays)
    fnr.fnr_cache_save(cache, str(tmp_path / "cache"))

    def image(c):
        fnr.fnr_render(ctx, c, [cam], p, rgba)
        torch.cuda.synchronize()
        return rgba.clone()

    calls = dict(render=lambda: fnr.fnr_render(ctx, cache, [cam], p, rgba),
                 build=lambda: fnr.fnr_build_cache(ctx, desc, *arrays),
                 build_mlp=lambda: fnr.fnr_build_cache_mlp(ctx, desc, *nets),
                 render_mlp=lambda: fnr.fnr_render_mlp(ctx, *nets, 8, cam, p, rgba),
                 load=lambda: fnr.fnr_cache_load(ctx, str(tmp_path / "cache")))

    def outcome(call_it):  # a cache is judged by what it renders
        c = call_it()
        torch.cuda.synchronize()
        got = rgba.clone() if c is None else image(c)
        if c is not None:
            fnr.fnr_cache_free(ctx, c)
        return got

    want = outcome(calls[call])
    rgba.zero_()
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    made, failed = [], []

    def under_another_context():
        other, primary, cur, dev = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_int()
        try:
            check(cu.cuDeviceGet(ctypes.byref(dev), 0))
            check(cu.cuDevicePrimaryCtxRetain(ctypes.byref(primary), dev))
            check(cu.cuCtxCreate_v2(ctypes.byref(other), 0, dev))  # and current on this thread
            try:
                # the runtime's switch itself, by a call that launches nothing: if it does not hold, go no further
                fnr.fnr_context_destroy(fnr.fnr_context_create(0, 0))
                check(cu.cuCtxGetCurrent(ctypes.byref(cur)))
                assert cur.value == primary.value
                check(cu.cuCtxSetCurrent(other))
                made.append(calls[call]())
                check(cu.cuCtxGetCurrent(ctypes.byref(cur)))
                assert cur.value == primary.value
            finally:
                check(cu.cuCtxDestroy_v2(other))
        except BaseException as e:
            failed.append(e)
        finally:
            if primary.value:
                cu.cuDevicePrimaryCtxRelease_v2(dev)

    t = threading.Thread(target=under_another_context)
    t.start()
    t.join()
    assert not failed, failed
    torch.cuda.synchronize()
    assert torch.equal(outcome(lambda: made[0]), want) if made[0] is not None else torch.equal(rgba, want)
    fnr.fnr_cache_free(ctx, cache)
