"""Split calls of disjoint stream ranges of one handle at the same time on two
streams, one with 16-byte rows and one without: each has its own arrival
counters, so outputs and states are those of the calls one after the other."""
from __future__ import annotations

import ctypes

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


N, ROWS, CALLS = 10_000, 2100, 12
# 16-byte rows of groups whose quarter indexes are first streams of the other
# range; rows that are not 16-byte aligned
RANGES = [((4000, 8000), 0), ((1, 3999), 2)]


def outputs():
    return [torch.zeros(ROWS * N + 8, dtype=torch.int32, device="cuda") for _ in RANGES]


@pytest.mark.parametrize("kind", [oracle.XOR128, oracle.MWC16X2, oracle.KISS_XOR])
def test_disjoint_ranges_on_two_streams(kind):
    log2 = ctypes.c_int()
    capi.check(capi.lib().gbrng_get_split(kind, ctypes.byref(log2)))
    g, h = Generator(kind, N, 17), Generator(kind, N, 17)
    got, want = outputs(), outputs()
    streams = [torch.cuda.Stream() for _ in RANGES]
    torch.cuda.synchronize()
    for _ in range(CALLS):
        for ((b, e), offset), out, s in zip(RANGES, got, streams):
            g.generate_range(b, e, ROWS, out, N, "u32", offset=offset, stream=s)
    torch.cuda.synchronize()
    capi.check(capi.lib().gbrng_set_split(kind, 0))  # whole calls, one stream
    try:
        for _ in range(CALLS):
            for ((b, e), offset), out in zip(RANGES, want):
                h.generate_range(b, e, ROWS, out, N, "u32", offset=offset)
    finally:
        capi.check(capi.lib().gbrng_set_split(kind, log2.value))
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert torch.equal(g.get_state(), h.get_state())
    g.close()
    h.close()


@pytest.mark.parametrize("kind", [oracle.MWC, oracle.KISS])
def test_jump_table_between_streams(kind):
    """MWC32 and KISS take the jumps from the handle's table: built by an aligned
    range's call on one stream, read by an unaligned one's on the other (equal
    segments), and rebuilt for another length while that may still be running."""
    log2 = ctypes.c_int()
    capi.check(capi.lib().gbrng_get_split(kind, ctypes.byref(log2)))
    g, h = Generator(kind, N, 18), Generator(kind, N, 18)
    got, want = outputs(), outputs()
    streams = [torch.cuda.Stream() for _ in RANGES]
    lengths = [2100, 1500, 2100, 900, 2100, 1500, 1200, 2100, 900, 1500, 2100, 1200]

    def calls(gen, outs, where):
        for rows in lengths:
            for ((b, e), offset), out, s in zip(RANGES, outs, where):
                gen.generate_range(b, e, rows, out, N, "u32", offset=offset, stream=s)

    torch.cuda.synchronize()
    calls(g, got, streams)
    torch.cuda.synchronize()
    capi.check(capi.lib().gbrng_set_split(kind, 0))
    try:
        calls(h, want, [None, None])
    finally:
        capi.check(capi.lib().gbrng_set_split(kind, log2.value))
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert torch.equal(g.get_state(), h.get_state())
    g.close()
    h.close()
