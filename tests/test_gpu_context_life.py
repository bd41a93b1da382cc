"""Making and destroying a context asks nothing of the rest of the device: it waits for no other stream and may happen
while a stream is being captured."""

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
    fnr.fnr_context_destroy(fnr.fnr_context_create(0, 0))
    return fnr


@pytest.mark.parametrize("layout", [0, 1])
def test_destroy_waits_for_no_other_stream(fnr, layout):
    import torch
    rng = np.random.default_rng(layout)
    k, D, l = 16, 2, 4
    src = tuple(torch.from_numpy(rng.random(n).astype(np.float32)).cuda() for n in (k ** 3, k ** 3 * 3 * D, l * l * D))
    ctx = fnr.fnr_context_create(0, 0)
    fnr.fnr_cache_free(ctx, fnr.fnr_build_cache(ctx, fnr.make_desc(k, D, l, 2, 1, layout=layout), *src))
    torch.cuda.synchronize()
    other = torch.cuda.Stream()
    with torch.cuda.stream(other):
        torch.cuda._sleep(1_000_000_000)  # half a second
    fnr.fnr_context_destroy(ctx)
    assert not other.query()
    other.synchronize()


def test_create_and_destroy_during_a_capture(fnr):
    import torch
    x = torch.zeros(64, device="cuda")
    x.add_(1)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        x.add_(1)
        fnr.fnr_context_destroy(fnr.fnr_context_create(0, 0))
        x.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert bool((x == 3).all())
