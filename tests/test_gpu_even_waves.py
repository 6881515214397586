"""Plain calls whose CTAs are made even (even_threads in
csrc/gen_kernels.cuh): calls of 77,824 to two million streams whose last wave
would be nearly empty, in every form of the rows (32-byte, 16-byte,
realigned with each tail), write what the same streams' blocks give in calls of
their own, and leave the same state."""
from __future__ import annotations

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import numpy as np  # noqa: E402
import oracle  # noqa: E402
from paper_1101_1846_gb300 import build, capi  # noqa: E402
from paper_1101_1846_gb300.generator import BatchItem, Generator, generate_batch  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


# just above one warp a scheduler; below and above whole waves of CTAs of 256,
# 512 and 1024 threads' groups; the ends of each form's tiles
STREAMS = [77_832, 77_828, 77_825, 86_016, 155_656, 172_035, 311_304, 360_004, 361_002, 622_600,
           700_001]


@pytest.mark.parametrize("n", STREAMS)
@pytest.mark.parametrize("kind", ["mwc", "xor128", "kiss"])
@pytest.mark.parametrize("fmt", ["u32", "f32"])
def test_even_calls_equal_batched_ones(kind, fmt, n):
    rows = 21
    g, h = Generator(kind, n, 9), Generator(kind, n, 9)
    out = torch.full((rows * n + 8,), -1, dtype=torch.int32, device="cuda")
    want = torch.full((rows * n,), -2, dtype=torch.int32, device="cuda")
    body = out[:rows * n].view(rows, n)
    for _ in range(2):  # the second pass starts from the states the first one left
        g.generate(rows, fmt, out=body.view(torch.float32) if fmt == "f32" else body)
        generate_batch([BatchItem(h, rows, want, 1 if fmt == "f32" else 0)])
        torch.cuda.synchronize()
        assert torch.equal(out[:rows * n], want)
        assert bool((out[rows * n:] == -1).all())


@pytest.mark.parametrize("n", STREAMS)
def test_even_xorshift8_equals_the_oracle(n):
    rows = 9
    g = Generator("xorshift8", n, 9)
    got = g.generate(rows, "u32").cpu().numpy().view(np.uint32).reshape(rows, n)
    pick = np.array(sorted({0, 1, 511, 512, 513, n // 2, n - 5, n - 4, n - 3, n - 2, n - 1}))
    st = oracle.seed_streams(oracle.XORSHIFT8, None, 9, pick)
    want, _ = oracle.generate(oracle.XORSHIFT8, None, st, rows, oracle.U32)
    assert np.array_equal(got[:, pick], np.asarray(want).view(np.uint32).reshape(rows, -1))


def test_a_callers_shape_stays():
    """A shape and a CTAs-per-SM choice that a caller set are used as they are
    and, set back, give way to the rule again; outputs never change."""
    import ctypes
    lib = capi.lib()
    n, rows = 360_000, 11
    want = Generator("kiss", n, 3).generate(rows, "u32")
    v, block, hint = (ctypes.c_int() for _ in range(3))
    capi.check(lib.gbrng_get_launch_class(oracle.KISS, 0, 0, v, block, hint))
    old = (v.value, block.value, hint.value)
    for shape in ((1, 64, 0), (2, 256, 1), old):
        capi.check(lib.gbrng_set_launch_class(oracle.KISS, 0, 0, *shape))
        assert torch.equal(Generator("kiss", n, 3).generate(rows, "u32"), want)
    for n in (360_004, 360_001):
        realigned = n % 2
        want = Generator("kiss", n, 3).generate(rows, "u32")
        for ctas in (0, 1):
            capi.check(lib.gbrng_set_row_ctas(oracle.KISS, 0, realigned, ctas))
            got = ctypes.c_int()
            capi.check(lib.gbrng_get_row_ctas(oracle.KISS, 0, realigned, got))
            assert got.value == ctas
            assert torch.equal(Generator("kiss", n, 3).generate(rows, "u32"), want)
