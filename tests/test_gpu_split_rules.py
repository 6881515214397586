"""Split calls against whole ones over the forms the segment rules choose
between: powers of two with and without the MWC table, equal lengths, one
wave, few threads, aligned, 16-byte and unaligned rows, and consumers."""
from __future__ import annotations

import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import Generator  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


class whole:
    """Runs a block with splitting off for `kind`."""

    def __init__(self, kind):
        self.kind, self.log2 = kind, ctypes.c_int()

    def __enter__(self):
        capi.check(capi.lib().gbrng_get_split(self.kind, ctypes.byref(self.log2)))
        capi.check(capi.lib().gbrng_set_split(self.kind, 0))

    def __exit__(self, *exc):
        capi.check(capi.lib().gbrng_set_split(self.kind, self.log2.value))


SHAPES = [(8, 130), (32, 129), (64, 5000), (4096, 1203), (12, 3001), (10_004, 2050),
          (20_000, 3001), (76_636, 1100), (40_001, 1100), (1003, 6001), (3000, 9001)]


@pytest.mark.parametrize("kind", range(6))
@pytest.mark.parametrize("n,rows", SHAPES)
def test_generate(kind, n, rows):
    a, b = Generator(kind, n, 40 + n), Generator(kind, n, 40 + n)
    for m in (rows, rows - 37):  # another length continues the streams
        got = a.generate(m)
        with whole(kind):
            want = b.generate(m)
        assert torch.equal(got, want), m
        assert torch.equal(a.get_state(), b.get_state()), m
        del got, want
    a.close()
    b.close()


@pytest.mark.parametrize("kind", range(6))
@pytest.mark.parametrize("n,rows", [(1, 5001), (64, 9000), (1003, 3333), (70_000, 1500)])
@pytest.mark.parametrize("op", ["sum_u32", "disc"])
def test_consumers(kind, n, rows, op):
    a, b = Generator(kind, n, 4), Generator(kind, n, 4)
    got = a.generate_reduce(rows, op)
    with whole(kind):
        want = b.generate_reduce(rows, op)
    assert torch.equal(got, want)
    assert torch.equal(a.get_state(), b.get_state())
    a.close()
    b.close()
