"""Whole disc calls of KISS_XOR choose the integer test or the FP32 blocks by
their CTAs: both sides of that line, lengths around the blocks, against the
generated outputs.  Whole numbers: exact."""
from __future__ import annotations

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import Generator  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


@pytest.mark.parametrize("n", [3, 152 * 256, 152 * 256 + 1, 76_636])
def test_whole_disc(n):
    g, h = Generator(oracle.KISS_XOR, n, 5), Generator(oracle.KISS_XOR, n, 5)
    for rows in (1, 2, 31, 32, 33, 129, 256):
        got = g.generate_reduce(rows, oracle.DISC)
        v = (h.generate(rows).long() & 0xFFFFFFFF) >> 8
        pairs = rows // 2
        want = (v[0:2 * pairs:2] ** 2 + v[1:2 * pairs:2] ** 2 < 1 << 48).sum(0)
        assert torch.equal(got, want), rows
        assert torch.equal(g.get_state(), h.get_state()), rows
    g.close()
    h.close()
