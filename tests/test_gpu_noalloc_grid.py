"""The grid of the allocation-free batched launch by what the list holds
(noalloc_ctas in csrc/batch.cu): few tiles with a long item, in cheap and in
costlier steps, and a tile per SM, against plain calls, bit for bit."""
from __future__ import annotations

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import BatchItem, Generator, _items  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


@pytest.mark.parametrize("kinds,fmt", [(("mwc", "xor128"), 0), (("mwc", "xor128"), 1),
                                       (("kiss",), 0)])
@pytest.mark.parametrize("count", [9, 300])
def test_grids_equal_plain_calls(kinds, fmt, count):
    rows, sizes = 384, [1 + 37 * i % 1500 for i in range(count)]
    gens, plain = ([Generator(kinds[i % len(kinds)], n, 3 + i) for i, n in enumerate(sizes)]
                   for _ in range(2))
    outs = [torch.full((rows * n + 1,), -1, dtype=torch.int32, device="cuda") for n in sizes]
    items = [BatchItem(g, rows, o[:-1], fmt) for g, o in zip(gens, outs)]
    torch.cuda.synchronize()
    capi.check(capi.lib().rng_generate_batch_noalloc(_items(items), count, None))
    torch.cuda.synchronize()
    for i, (p, o) in enumerate(zip(plain, outs)):
        assert torch.equal(o[:-1], p.generate(rows, fmt).view(torch.int32).reshape(-1)), i
        assert int(o[-1]) == -1
