"""Jumps by the composed matrix (xor128, XORSHIFT8) and by the CTA's tables
(KISS kinds): set-bit counts on both sides of every batch of matrices, and
more streams than the resident threads, against the oracle."""
from __future__ import annotations

import random

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


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


def state_of(g: Generator) -> np.ndarray:
    return g.get_state().numpy().view(np.uint32).T


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("bits", [1, 2, 3, 4, 5, 8, 15, 16, 17, 33, 63, 64])
def test_set_bits(kind, bits):
    n = 1003
    rng = random.Random(bits)
    idx = np.array([0, 1, 31, 32, 511, 512, n - 1])
    a = oracle.multipliers_for(kind, n)
    a = a if a is None else a[idx]
    st = oracle.seed_streams(kind, a, 11, idx)
    g = Generator(kind, n, 11)
    for _ in range(2):
        k = sum(1 << b for b in rng.sample(range(64), bits))
        g.jump(k)
        st = oracle.jump_streams(kind, a, st, k)
        assert np.array_equal(state_of(g)[idx], st[:, :g.words]), k
    g.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("k", [1, 2, 3, 65, 4097])
def test_equals_single_steps(kind, k):
    n = 130
    g, h = Generator(kind, n, 8), Generator(kind, n, 8)
    g.jump(k)
    h.generate(k)
    assert torch.equal(g.get_state(), h.get_state())
    g.close()
    h.close()


@pytest.mark.parametrize("kind", [oracle.XOR128, oracle.XORSHIFT8])
@pytest.mark.parametrize("n", [1, 511, 513, 400_001])
def test_stream_counts(kind, n):
    k = 0x0123456789ABCDEF
    g = Generator(kind, n, 5)
    idx = np.unique(np.array([0, 1, n // 2, 152 * 3 * 512 - 1, 152 * 3 * 512, n - 2, n - 1])
                    .clip(0, n - 1))
    st = oracle.seed_streams(kind, None, 5, idx)
    g.jump(k)
    want = oracle.jump_streams(kind, None, st, k)
    assert np.array_equal(state_of(g)[idx], want[:, :g.words])
    g.close()
