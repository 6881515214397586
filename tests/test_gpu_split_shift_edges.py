"""Unaligned split calls at the edges of their CTAs (125 groups of four, spread
evenly): group counts on both sides of one and two CTAs with every tail, tails
alone, every kind and every cycle of row alignments, against whole calls, with the
words around the output.  Each case is checked to be split."""
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

SHIFTED = 1  # SplitForm in csrc/gbrng.cuh


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


def check(kind, n, rows, fmt, ld, offset):
    lib = capi.lib()
    wanted = lib._ZN5gbrng12split_wantedEiNS_9SplitFormEimm
    wanted.restype = ctypes.c_bool
    wanted.argtypes = [ctypes.c_int] * 3 + [ctypes.c_uint64] * 2
    assert wanted(kind, SHIFTED, fmt, n, rows)
    log2 = ctypes.c_int()
    capi.check(lib.gbrng_get_split(kind, ctypes.byref(log2)))
    words = offset + (rows - 1) * ld + n
    results = []
    for split in (True, False):
        if not split:
            capi.check(lib.gbrng_set_split(kind, 0))
        try:
            g = Generator(kind, n, 61)
            out = torch.full((words + 9,), -7, dtype=torch.int32, device="cuda")
            for _ in range(2):
                g.generate_range(0, n, rows, out, ld, fmt, offset=offset)
            results.append((out, g.get_state()))
            g.close()
        finally:
            capi.check(lib.gbrng_set_split(kind, log2.value))
    (got, state), (want, state_whole) = results
    assert torch.equal(got, want)
    assert torch.equal(state, state_whole)


KINDS = [oracle.MWC, oracle.XOR128, oracle.KISS, oracle.MWC16X2, oracle.XORSHIFT8,
         oracle.KISS_XOR]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("groups", [124, 125, 126, 250, 251])
@pytest.mark.parametrize("tail", [0, 1, 2, 3])
def test_groups_and_tails(kind, groups, tail):
    n = 4 * groups + tail
    check(kind, n, 1301, tail & 1, n + (0 if tail else 1), 0)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("dr,offset", [(0, 1), (0, 2), (0, 3), (1, 0), (2, 1), (3, 0)])
def test_row_cycles(kind, dr, offset):
    check(kind, 301, 1303, dr & 1, 304 + dr, offset)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [1, 2, 3])
def test_tails_alone(kind, n):
    check(kind, n, 7001, n & 1, n + 1, 1)
