"""A batch holds its plans' memory and a work list, not a second copy of the Jacobi's operands."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2204_12879_gb300 import lrstv
    return lrstv


def test_batch_memory_is_its_plans(L):
    """Three cubes whose operands (92 MB each) would show; the work list and queue of 369 slices, the allocations' rounding to
    2 MiB each and the stream stay below 16 MB."""
    import torch
    shapes = [(200, 200, 80)] * 3
    params = [L.Params.make(200, 200, max_iter=2, flags=L.FLAG_WARM_START) for _ in shapes]
    with L.Batch([(16, 16, 4)], [L.Params.make(16, 16, max_iter=1)]) as b:  # the context's own first allocations
        b.run([torch.rand(16 * 16 * 4, device="cuda")])
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    with L.Batch(shapes, params) as b:
        torch.cuda.synchronize()
        held = before - torch.cuda.mem_get_info()[0]
        plans = sum(b.plan(i).nbytes for i in range(3))
    print("held", held, "plans", plans)
    assert held <= plans + (16 << 20)


def test_a_lent_plan_can_still_step(L):
    """The batch and a plan it lends use the same operands, one after the other."""
    import torch
    shape = (40, 36, 6)
    prm = L.Params.make(40, 36, max_iter=4, flags=L.FLAG_WARM_START)
    ys = [torch.rand(40 * 36 * 6, generator=torch.Generator().manual_seed(s)).cuda() for s in (1, 2)]
    with L.Plan(*shape, prm) as p:
        p.init(ys[0])
        p.iterate(5)
        want = p.get("L")
    with L.Batch([shape, shape], [prm, prm]) as b:
        b.init(ys)
        b.iterate(4)
        b.plan(0).iterate(1)
        assert torch.equal(b.plan(0).get("L"), want)
