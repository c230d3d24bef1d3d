"""What a sort of product records does to its stream."""
import pytest
import torch

from paper_2301_07684_gb300 import sfq
from paper_2301_07684_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("n", [2, 1000, 16384, 16385])
def test_earlier_work_has_finished_on_return(n, noalloc):
    """A sort of any size synchronises its stream once before it moves records."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=4)
    out = sfq.ProductBuffers(n, ctx.dtype, "cuda")
    out.parent_id[:] = torch.arange(n, 0, -1, device="cuda")
    scratch = torch.empty(sfq.sort_scratch_bytes(n), dtype=torch.uint8, device="cuda")
    for t in (out.px, out.py, out.pz, out.step, out.meta):
        t.zero_()
    sort = (lambda: ctx.sort_products_noalloc(out, n)) if noalloc else (lambda: ctx.sort_products(out, n, scratch))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        sort()                                             # loads the kernels
        for _ in range(2):
            torch.cuda._sleep(20000000)                    # about 10 ms
            queued = torch.cuda.Event()
            queued.record(s)
            assert not queued.query()
            sort()
            assert queued.query()
    torch.cuda.synchronize()
    assert torch.equal(out.parent_id, torch.arange(1, n + 1, device="cuda"))


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("n", [2, 16384, 16385])
def test_a_sort_is_refused_under_capture(n, noalloc):
    """A sort is not recorded into a graph: it returns an error, moves nothing and leaves the
    capture as it was."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=4)
    out = sfq.ProductBuffers(n, ctx.dtype, "cuda")
    given = torch.arange(n, 0, -1, device="cuda")
    out.parent_id.copy_(given)
    for t in (out.px, out.py, out.pz, out.step, out.meta):
        t.zero_()
    scratch = torch.empty(sfq.sort_scratch_bytes(n), dtype=torch.uint8, device="cuda")
    sort = (lambda: ctx.sort_products_noalloc(out, n)) if noalloc else (lambda: ctx.sort_products(out, n, scratch))
    sort()
    out.parent_id.copy_(given)
    mark = torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mark.add_(1)
        with pytest.raises(sfq.SfqError):
            sort()
        mark.add_(1)
    assert torch.equal(out.parent_id, given)
    graph.replay()
    torch.cuda.synchronize()
    assert float(mark) == 2.0 and torch.equal(out.parent_id, given)
    sort()
    assert torch.equal(out.parent_id, given.flip(0))
