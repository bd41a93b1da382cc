"""Brick builds from device arrays on a stream that has work queued ahead of them: what the build reads on the host
(the direction-bin tables) lives until the stream has got there, and a build that fails returns with nothing of it
still queued."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K, D = 24, 4


@pytest.fixture(scope="module")
def fnr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    torch.cuda.set_device(0)
    yield fnr
    fnr.fnr_testing_fail_allocations(0, 0)


def arrays(l):
    import torch
    rng = np.random.default_rng(l)
    dev = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()
    return (dev(np.where(rng.random(K ** 3) < 0.02, 5.0, 0.0)), dev(rng.standard_normal(K ** 3 * 3 * D)),
            dev(rng.standard_normal(l * l * D)))


def busy_stream():
    import torch
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(100_000_000)  # 50 ms
    return s


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("l", [2, 5, 700, 2500])
def test_tables_behind_queued_work(fnr, l, prec):
    import torch

    def table(ptr):
        class _V:
            __cuda_array_interface__ = {"shape": (l,), "typestr": "<f4", "data": (ptr, False), "version": 3}
        return torch.as_tensor(_V(), device="cuda").cpu().numpy()

    src = arrays(l)
    torch.cuda.synchronize()
    ctx = fnr.fnr_context_create(0, 0)
    try:
        got = []
        for layout, stream in ((fnr.FNR_LAYOUT_DENSE, None), (fnr.FNR_LAYOUT_BRICKS, busy_stream())):
            c = fnr.fnr_build_cache(ctx, fnr.make_desc(K, D, l, prec, layout=layout), *src, stream=stream)
            lay = fnr.fnr_cache_get_layout(c)
            got.append((table(lay.cos_theta_dev), table(lay.phi_key_dev)))
        assert np.array_equal(got[0], got[1])
        assert np.allclose(got[1][0], np.cos(np.arange(l) * np.pi / l), atol=1e-7)
    finally:
        fnr.fnr_context_destroy(ctx)


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_failed_build_leaves_nothing_queued(fnr, prec):
    import torch
    src = arrays(8)
    torch.cuda.synchronize()
    desc = fnr.make_desc(K, D, 8, prec, layout=fnr.FNR_LAYOUT_BRICKS)
    ctx = fnr.fnr_context_create(0, 1 << 30)
    try:
        for i in range(16):
            stream = busy_stream()
            fnr.fnr_testing_fail_allocations(i, 1)
            try:
                c = fnr.fnr_build_cache(ctx, desc, *src, stream=stream)
            except fnr.FnrError as e:
                assert e.status == fnr.FNR_ERR_OOM
                # the first allocation is made before anything is queued
                assert i == 0 or stream.query(), f"allocation {i}"
                assert fnr.fnr_context_used_bytes(ctx) == 0
                continue
            finally:
                fnr.fnr_testing_fail_allocations(0, 0)
            break
        else:
            raise AssertionError("the build kept allocating")
        assert i >= 4  # the stage, the brick ranks, the cache and the slots at least
        fnr.fnr_cache_free(ctx, c)
    finally:
        fnr.fnr_context_destroy(ctx)
