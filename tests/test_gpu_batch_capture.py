"""GPU: a batch refuses a stream that is being captured, leaves the capture as it was, and works afterwards; a refused
call leaves none of its pointers behind."""
import pytest

torch = pytest.importorskip("torch")

import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("called_before", (False, True))
def test_capture_is_refused(called_before):
    import paper_2204_06666_gb300 as eh
    mats = [gen.tet_lap3d(N=n) for n in (8, 12)]
    plans = [eh.Plan(A) for A in mats]
    B = eh.Batch(plans)
    xs = [torch.from_numpy(gen.uniform(A.n, 3 + i)).cuda() for i, A in enumerate(mats)]
    ys, refs = ([torch.zeros_like(x) for x in xs] for _ in range(2))
    for P, x, y in zip(plans, xs, refs):
        P.spmv(x, y)
    if called_before:
        B.spmv(xs, [torch.zeros_like(x) for x in xs])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    other = torch.zeros_like(xs[0])
    with torch.cuda.graph(g):
        with pytest.raises(eh.EhybError):
            B.spmv(xs, ys)
        plans[0].spmv(xs[0], other)      # a product can be captured
    assert not any(y.any() for y in ys)
    B.spmv(xs, ys)
    assert all(torch.equal(y, r) for y, r in zip(ys, refs))
    g.replay()
    assert torch.equal(other, refs[0])


def test_refused_pointers_do_not_stay():
    import paper_2204_06666_gb300 as eh
    mats = [gen.tet_lap3d(N=n) for n in (8, 12)]
    plans = [eh.Plan(A) for A in mats]
    B = eh.Batch(plans)
    xs = [torch.from_numpy(gen.uniform(A.n, 3 + i)).cuda() for i, A in enumerate(mats)]
    ys = [torch.zeros_like(x) for x in xs]
    B.spmv(xs, ys)
    first = [torch.zeros_like(xs[0]), ys[1]]
    with pytest.raises(eh.EhybError):
        B.spmv(xs, [first[0], xs[1]])    # x and y of the second are one array
    B.spmv(xs, first)
    assert torch.equal(first[0], ys[0])
