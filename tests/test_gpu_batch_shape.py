"""The shapes that plans choose by what they hold (choose_shape and
refill_shape in csrc/batch.cu): lists on both sides of each line of the rules,
launched, refilled and through the allocation-free entry point, give what
plain calls of the same generators give, bit for bit."""
from __future__ import annotations

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import BatchItem, Generator, Plan, _items  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


KINDS = ("mwc", "xor128", "kiss")


class Lists:
    """One generator per item with its plain twin; take() makes a list."""

    def __init__(self, sizes):
        self.gens = [Generator(KINDS[i % 3], n, 5 + i) for i, n in enumerate(sizes)]
        self.plain = [Generator(KINDS[i % 3], n, 5 + i) for i, n in enumerate(sizes)]

    def take(self, rows, pick=None):
        pick = range(len(self.gens)) if pick is None else pick
        self.outs = [(i, torch.full((rows * self.gens[i].n_streams + 1,), -1, dtype=torch.int32,
                                    device="cuda")) for i in pick]
        self.rows = rows
        return [BatchItem(self.gens[i], rows, o[:-1], i % 2) for i, o in self.outs]

    def check(self):
        torch.cuda.synchronize()
        for i, o in self.outs:
            want = self.plain[i].generate(self.rows, i % 2).view(torch.int32).reshape(-1)
            assert torch.equal(o[:-1], want), i
            assert int(o[-1]) == -1


def sizes_of(tiles):
    """Streams per item for `tiles` tiles of 128 threads: odd and even
    remainders in front, then one item of whole tiles."""
    small = [1, 3, 4, 131, 255, 256, 257, 500, 505, 508]
    # a tile each, but 505 two (500 streams, then 4 with the tail)
    return small + [512 * (tiles - len(small) - 1)]


@pytest.mark.parametrize("per_sm,over,rows,shape", [
    (0, 30, 383, (128, 2)), (0, 30, 384, (64, 2)),
    (8, 0, 384, (64, 2)), (8, 1, 384, (128, 2)), (8, 0, 20, (128, 2)), (8, 1, 20, (512, 1)),
    (13, 0, 384, (128, 2)), (13, 1, 384, (512, 1))])
def test_shapes_equal_plain_calls(per_sm, over, rows, shape):
    sm = sms()
    x = Lists(sizes_of(per_sm * sm + over))
    plan = Plan(x.take(rows))
    assert plan.shape == (shape[0], sm * shape[1])
    plan.launch()
    x.check()


def test_refills_choose_their_shape():
    sm = sms()
    x = Lists(sizes_of(13 * sm + 1))
    plan = Plan(x.take(17, range(10)))
    assert plan.shape == (128, 2 * sm)
    plan.launch()
    x.check()
    for rows, pick, threads in ((127, range(10), 512), (128, range(10), 128), (9, None, 512),
                                (385, range(10), 128), (130, None, 512), (4, [1], 512)):
        plan.refill(x.take(rows, pick))
        assert plan.shape == (threads, sm)
        plan.launch()
        x.check()


@pytest.mark.parametrize("over,threads", [(0, 128), (1, 512)])
def test_refill_tile_line(over, threads):
    x = Lists(sizes_of(5 * sms() + over))
    plan = Plan(x.take(3))
    plan.launch()
    x.check()
    plan.refill(x.take(128))
    assert plan.shape == (threads, sms())
    plan.launch()
    x.check()


def test_explicit_shapes_stay():
    x = Lists(sizes_of(40))
    plan = Plan(x.take(5), threads=256, ctas_per_sm=2)
    before = plan.shape
    assert before == (256, 2 * sms())
    plan.launch()
    x.check()
    plan.refill(x.take(400))
    assert plan.shape == before
    plan.launch()
    x.check()


@pytest.mark.parametrize("per_sm,rows", [(0, 383), (0, 384), (8, 384), (9, 20)])
def test_noalloc_grids_equal_plain_calls(per_sm, rows):
    x = Lists(sizes_of(per_sm * sms() + 30))
    items = x.take(rows)
    torch.cuda.synchronize()
    capi.check(capi.lib().rng_generate_batch_noalloc(_items(items), len(items), None))
    x.check()
