"""The battery's sample kernel at its edges (columns per pass, rows in no
sample, full buckets, many candidates, the cap), against the oracle or plain
PyTorch counts.  Whole numbers: every comparison is exact."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1101_1846_gb300 import battery, build, capi  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    capi.lib()


def check(u: np.ndarray):
    rows, n = u.shape
    u = np.ascontiguousarray(u)
    c = battery.counts(torch.from_numpy(u.view(np.int32)).cuda(), n, rows)
    o = oracle.battery_counts(u)
    assert c["ones"] == o["ones"] and c["birthday_samples"] == o["birthday_samples"]
    for k in ("bytes", "serial", "birthday"):
        assert np.array_equal(c[k], o[k]), k


def random_words(rng, rows: int, n: int) -> np.ndarray:
    return rng.integers(0, 1 << 32, size=(rows, n), dtype=np.uint64).astype(np.uint32)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 5000])
@pytest.mark.parametrize("rows", [511, 512, 513, 1539])
def test_columns_and_rows(n, rows):
    check(random_words(np.random.Generator(np.random.PCG64(n * rows)), rows, n))


@pytest.mark.parametrize("k", [14, 15, 16, 17, 255, 256, 512])
def test_days_in_one_bucket(k):
    """k days of each sample share their top 10 bits."""
    rng = np.random.Generator(np.random.PCG64(k))
    u = random_words(rng, 512, 40)
    u[:k] = (u[:k] & np.uint32((1 << 22) - 1)) | np.uint32(617 << 22)
    check(rng.permuted(u, axis=0))


@pytest.mark.parametrize("k", [1, 30, 31, 32, 33, 34, 200, 500])
def test_equal_spacings(k):
    """k spacings of each sample are equal (k - 1 repeats or a few more)."""
    rng = np.random.Generator(np.random.PCG64(100 + k))
    cols = []
    for _ in range(20):
        gaps = np.concatenate([np.full(k, 30000), rng.choice(np.arange(20000, 30000), 512 - k,
                                                             replace=False)])
        days = np.cumsum(rng.permutation(gaps)).astype(np.uint32)
        cols.append((rng.permutation(days) << np.uint32(8)) | np.uint32(rng.integers(0, 256)))
    check(np.stack(cols, axis=1))


@pytest.mark.parametrize("word", [0, 0xFFFFFFFF, 0x12345678])
def test_constant_words(word):
    check(np.full((1024, 19), word, dtype=np.uint32))


def test_past_the_cap():
    """2^21 samples end inside the second block: the streams past them and
    the rows after the block are counted, but make no sample."""
    n, rows = (1 << 20) + 8, 1030
    u = torch.randint(-2**31, 2**31, (rows, n), dtype=torch.int32, device="cuda",
                      generator=torch.Generator("cuda").manual_seed(3))
    c = battery.counts(u, n, rows)
    assert c["birthday_samples"] == capi.RNG_BATTERY_BIRTHDAY_MAX
    bytes_ = torch.zeros(256, dtype=torch.int64, device="cuda")
    serial = torch.zeros(256, dtype=torch.int64, device="cuda")
    ones = 0
    for r in range(0, rows, 10):
        x = u[r:r + 10].long() & 0xFFFFFFFF
        bytes_ += torch.bincount((x >> 24).flatten(), minlength=256)
        serial += torch.bincount(((x[0::2] >> 28) * 16 + (x[1::2] >> 28)).flatten(),
                                 minlength=256)
        ones += sum(int(((x >> b) & 1).sum()) for b in range(32))
    assert c["ones"] == ones
    assert np.array_equal(c["bytes"], bytes_.cpu().numpy().astype(np.uint64))
    assert np.array_equal(c["serial"], serial.cpu().numpy().astype(np.uint64))
    cut = capi.RNG_BATTERY_BIRTHDAY_MAX - n
    first = battery.counts(u[:512].contiguous(), n, 512)
    second = battery.counts(u[512:1024, :cut].contiguous(), cut, 512)
    assert np.array_equal(c["birthday"], first["birthday"] + second["birthday"])
