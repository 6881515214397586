"""A plan's captured launch after a refill: replaying it runs the new list, for
plans whose first list chose each shape, and for a plan refilled before the
capture.  Outputs against plain calls of the same generators, bit for bit."""
from __future__ import annotations

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import BatchItem, Generator, Plan  # noqa: E402

KINDS = ("mwc", "xor128", "kiss")
SMALL = [1, 3, 131, 505, 508, 2268, 4000]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


@pytest.mark.parametrize("before", [False, True])
@pytest.mark.parametrize("sizes,rows,threads", [
    (SMALL, 400, 64), (SMALL, 21, 128), (SMALL + [1_100_000], 21, 512)])
def test_replay_after_refill(sizes, rows, threads, before):
    gens = [Generator(KINDS[i % 3], n, 70 + i) for i, n in enumerate(sizes)]
    plain = [Generator(KINDS[i % 3], n, 70 + i) for i, n in enumerate(sizes)]

    def take():
        outs = [torch.full((rows * n + 1,), -1, dtype=torch.int32, device="cuda") for n in sizes]
        return outs, [BatchItem(g, rows, o[:-1], i % 2) for i, (g, o) in enumerate(zip(gens, outs))]

    first, items = take()
    plan = Plan(items)
    assert plan.shape[0] == threads
    if before:
        plan.refill(items)
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        plan.launch(side)
    held = plan.shape, plan.tiles
    for _ in range(2):
        outs, items = take()
        plan.refill(items)
        assert (plan.shape, plan.tiles) == held
        graph.replay()
        torch.cuda.synchronize()
        for i, (p, o) in enumerate(zip(plain, outs)):
            assert torch.equal(o[:-1], p.generate(rows, i % 2).view(torch.int32).reshape(-1)), i
            assert int(o[-1]) == -1
    assert all(bool((o == -1).all()) for o in first)
    plan.close()
