"""Split calls whose rows are not 16-byte aligned (odd stream counts, offset
outputs, ranges): outputs, states and the words around the output against
the oracle, bit for bit."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import Generator  # noqa: E402

SPLIT = [oracle.MWC, oracle.XOR128, oracle.KISS, oracle.MWC16X2, oracle.KISS_XOR]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


def state_of(g: Generator) -> np.ndarray:
    return g.get_state().numpy().view(np.uint32).T


def run(kind, n, steps, fmt, offset=0, s_begin=0, s_end=None, ld=None, calls=1):
    s_end = n if s_end is None else s_end
    count, ld = s_end - s_begin, n if ld is None else ld
    a = oracle.multipliers_for(kind, n)
    st = oracle.seed_streams(kind, a, 31 + n, np.arange(n))
    g = Generator(kind, n, 31 + n)
    words = (steps - 1) * ld + count
    for _ in range(calls):
        buf = torch.full((offset + words + 9,), -7, dtype=torch.int32, device="cuda")
        g.generate_range(s_begin, s_end, steps, buf, ld, fmt, offset=offset)
        got = buf.cpu().numpy()
        exp, new = oracle.generate(kind, None if a is None else a[s_begin:s_end],
                                   st[s_begin:s_end], steps, fmt)
        st[s_begin:s_end] = new
        want = np.full_like(got, -7)
        rows = np.lib.stride_tricks.as_strided(want[offset:], (steps, count), (4 * ld, 4))
        rows[:] = np.ascontiguousarray(exp).view(np.int32)
        assert np.array_equal(got, want)
        assert np.array_equal(state_of(g), st[:, :g.words])
    g.close()


@pytest.mark.parametrize("kind", SPLIT)
@pytest.mark.parametrize("fmt", [oracle.U32, oracle.F32])
@pytest.mark.parametrize("n,steps", [(1, 3001), (3, 2048), (5, 1030), (127, 1027), (129, 1500),
                                     (997, 1026), (1001, 2049), (4999, 1031)])
def test_odd_streams(kind, fmt, n, steps):
    run(kind, n, steps, fmt, calls=2)


@pytest.mark.parametrize("kind", SPLIT)
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_offset_outputs(kind, offset):
    run(kind, 512, 1100, oracle.U32, offset=offset)


@pytest.mark.parametrize("kind", SPLIT)
@pytest.mark.parametrize("s_begin,s_end,ld,offset", [(0, 4, 12, 1), (3, 500, 497, 0),
                                                     (5, 130, 1001, 2), (700, 703, 3, 3),
                                                     (1, 1000, 1002, 0)])
def test_ranges(kind, s_begin, s_end, ld, offset):
    run(kind, 1001, 1300, oracle.F32, offset, s_begin, s_end, ld)


@pytest.mark.parametrize("kind", SPLIT)
def test_split_equals_whole(kind):
    """Group counts on both sides of a CTA's 249, whole calls as the reference."""
    log2 = ctypes.c_int()
    capi.check(capi.lib().gbrng_get_split(kind, ctypes.byref(log2)))
    for n in (995, 996 + 2, 1000 + 1, 1993, 60_003):
        a, b = Generator(kind, n, 5), Generator(kind, n, 5)
        got = a.generate(777)
        capi.check(capi.lib().gbrng_set_split(kind, 0))
        try:
            want = b.generate(777)
        finally:
            capi.check(capi.lib().gbrng_set_split(kind, log2.value))
        assert torch.equal(got, want), n
        assert torch.equal(a.get_state(), b.get_state()), n
        a.close()
        b.close()


@pytest.mark.parametrize("kind", [oracle.MWC, oracle.KISS])
def test_captured_in_a_graph(kind):
    n, steps = 251, 1024
    a = oracle.multipliers_for(kind, n)
    st = oracle.seed_streams(kind, a, 9, np.arange(n))
    g = Generator(kind, n, 9)
    out = torch.empty((steps, n), dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        g.generate(steps, out=out)
    for _ in range(2):
        graph.replay()
        exp, st = oracle.generate(kind, a, st, steps, oracle.U32)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), exp)
    g.close()
