"""Which generate calls are split into jumped segments (split_wanted in
csrc/generate.cu), on the CPU: calls on both sides of the lines of the rule, by
kind, form of the rows, streams and rows."""
from __future__ import annotations

import ctypes

import pytest

from paper_1101_1846_gb300 import build, capi

MWC, XOR128, KISS, MWC16X2, XORSHIFT8, KISS_XOR = range(6)
ALIGNED, SHIFTED, ROWS16 = range(3)


U32, F32 = range(2)


@pytest.fixture(scope="module")
def wanted():
    build.build()
    # gbrng::split_wanted(int kind, SplitForm, int fmt, uint64_t, uint64_t)
    fn = capi.lib()._ZN5gbrng12split_wantedEiNS_9SplitFormEimm
    fn.restype = ctypes.c_bool
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_uint64, ctypes.c_uint64]
    return fn


@pytest.mark.parametrize("kind,form,fmt,streams,whole,split", [
    (XOR128, SHIFTED, U32, 1, 1118, 4400), (XOR128, SHIFTED, F32, 3, 2500, 2800),
    (XORSHIFT8, SHIFTED, F32, 3, 4000, 7000), (KISS_XOR, SHIFTED, U32, 3, 260, 560),
    (KISS_XOR, SHIFTED, F32, 3, 300, 360), (MWC, SHIFTED, F32, 2, 313, 450),
    (KISS, SHIFTED, U32, 1, 500, 600), (KISS, SHIFTED, F32, 1, 300, 380),
    (MWC16X2, SHIFTED, U32, 3, 400, 450),
    (XORSHIFT8, SHIFTED, U32, 4, 1254, 1300), (KISS, SHIFTED, U32, 4, 256, 288),
    (KISS, SHIFTED, F32, 4, 255, 256), (KISS_XOR, SHIFTED, U32, 4, 160, 200),
    (KISS_XOR, SHIFTED, U32, 5, 128, 129), (KISS, SHIFTED, U32, 1001, 255, 256),
    (KISS_XOR, ROWS16, U32, 76_636, 192, 320), (KISS_XOR, ALIGNED, U32, 76_632, 400, 1600),
    (KISS_XOR, ALIGNED, U32, 4096, 160, 180), (MWC16X2, ALIGNED, U32, 60_000, 500, 1000),
    (MWC16X2, ALIGNED, U32, 64, 160, 180), (KISS, ROWS16, U32, 76_636, 200, 500),
    (MWC, ALIGNED, U32, 76_632, 400, 500), (KISS, ALIGNED, U32, 202_048, 150, 160),
    (KISS, ROWS16, U32, 202_044, 150, 1156), (MWC, ALIGNED, F32, 90_000, 200, 300),
    (MWC16X2, ROWS16, F32, 76_636, 200, 497),
    (XOR128, ALIGNED, F32, 14_472, 400, 927), (XOR128, ROWS16, F32, 1004, 300, 400),
    (XOR128, ALIGNED, U32, 64, 399, 400), (XOR128, ALIGNED, F32, 4, 299, 300),
    (XOR128, ALIGNED, U32, 1000, 700, 760), (XOR128, ALIGNED, U32, 20_000, 1024, 1500),
    (XORSHIFT8, ALIGNED, U32, 76_632, 16_000, 24_000),
    (XORSHIFT8, ALIGNED, U32, 50_000, 8000, 16_000),
    (XORSHIFT8, ALIGNED, F32, 8, 1023, 1024),
    (XORSHIFT8, ALIGNED, U32, 4096, 1100, 1150)])
def test_lines(wanted, kind, form, fmt, streams, whole, split):
    assert not wanted(kind, form, fmt, streams, whole)
    assert wanted(kind, form, fmt, streams, split)
    assert not wanted(kind, form, fmt, (1 << 19) + 4, split)  # enough streams as they are
