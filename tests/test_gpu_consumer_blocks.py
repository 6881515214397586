"""The consumers' blocks: lengths around the blocks of 16 pairs and 256
outputs against the oracle, and enough pairs that some hundred blocks hold a
point too near the circle for the FP32 test.  Whole numbers: exact."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import Generator  # noqa: E402

KINDS = [oracle.MWC, oracle.XOR128, oracle.KISS, oracle.MWC16X2, oracle.XORSHIFT8,
         oracle.KISS_XOR]
OPS = [oracle.SUM_U32, oracle.SUM_U24, oracle.DISC]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("op", OPS)
def test_lengths(kind, op):
    n = 517
    a = oracle.multipliers_for(kind, n)
    st = oracle.seed_streams(kind, a, 21, np.arange(n))
    g = Generator(kind, n, 21)
    for steps in (1, 2, 31, 32, 33, 34, 64, 65, 255, 256, 257, 511, 512, 1025):
        got = g.generate_reduce(steps, op).cpu().numpy().view(np.uint64)
        exp, st = oracle.reduce(kind, a, st, steps, op)
        assert np.array_equal(got, exp), steps
        assert np.array_equal(g.get_state().numpy().view(np.uint32).T, st[:, :g.words]), steps
    g.close()


@pytest.mark.parametrize("kind", [oracle.MWC, oracle.XOR128, oracle.KISS])
def test_points_near_the_circle(kind):
    n, rows = 1 << 18, 1024
    g, h = Generator(kind, n, 77), Generator(kind, n, 77)
    got = g.generate_reduce(rows, oracle.DISC)
    want = torch.zeros(n, dtype=torch.int64, device="cuda")
    near = 0
    for _ in range(rows // 128):
        v = (h.generate(128).long() & 0xFFFFFFFF) >> 8
        r = v[0::2] ** 2 + v[1::2] ** 2 - (1 << 48)
        want += (r < 0).sum(0)
        near += int((r.abs() < 1 << 27).sum())
    # |d| < 2^43 in the scale of the outputs' squares: a ring of width 2^-20 in
    # x^2 + y^2 holds pi/4 2^-20 of the points, 100.5 expected here
    assert near > 50
    assert torch.equal(got, want)
    g.close()
    h.close()
