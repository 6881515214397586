"""Refilled plans on the CPU: the library's plan code over stand-ins for the
CUDA runtime's calls (native/refill_check.cu).  A launch that was captured
before a refill of as many tiles covers every stream of the new list once, with
the CTA size it was captured with, and touches no record of the old list."""
from __future__ import annotations

import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]
SMS = 152


@pytest.fixture(scope="module")
def refill_bin(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not Path(nvcc).exists():
        pytest.skip("nvcc not found")
    out = tmp_path_factory.mktemp("refill") / "refill_check"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                    "-I", str(ROOT / "include"), "-I", str(ROOT / "paper_1101_1846_gb300" / "csrc"),
                    "-o", str(out), str(ROOT / "tests" / "native" / "refill_check.cu")],
                   check=True, capture_output=True, timeout=600)
    return out


def run(refill_bin, before, rows, sizes):
    text = f"{before} {rows} {len(sizes)}\n" + "\n".join(map(str, sizes)) + "\n"
    r = subprocess.run([str(refill_bin)], input=text, capture_output=True, text=True, check=True,
                       timeout=120)
    captured, after, allocs, *records = r.stdout.strip().split("\n")
    return captured, after, int(allocs.split()[1]), [tuple(map(int, x.split())) for x in records]


# few tiles of long and of short items, and lists on both sides of the lines
# between the shapes that plans and refills choose
LISTS = [(400, [2268, 1001, 8, 3, 131]), (1018, [2268] * 216), (20, [505] * 40),
         (200, [43_000] * 9), (384, [512 * 9 * SMS]), (20, [512 * 9 * SMS, 7]),
         (130, [512 * 5 * SMS, 9]), (256, [65_536] * 64)]


@pytest.mark.parametrize("before", [0, 1])
@pytest.mark.parametrize("rows,sizes", LISTS)
def test_captured_launch_replays_the_new_list(refill_bin, before, rows, sizes):
    captured, after, _, records = run(refill_bin, before, rows, sizes)
    assert after == captured
    seen = {}
    for item, _, s0, streams, new in records:
        assert new, "a record of the old list"
        seen.setdefault(item, []).append((s0, streams))
    for i, n in enumerate(sizes):
        at = 0
        for s0, streams in sorted(seen[i]):
            assert s0 == at, (i, s0, at)
            at += streams
        assert at == n, (i, at)


@pytest.mark.parametrize("rows,sizes,fewer,more_rows", [
    (256, [65_536] * 12, 5, 400), (20, [512 * 9 * SMS], 1, 400), (17, [512 * 5 * SMS, 7], 2, 130),
    (1018, [2268] * 216, 216, 20)])
def test_a_list_that_does_not_outgrow_the_first_allocates_nothing(refill_bin, rows, sizes, fewer,
                                                                  more_rows):
    """The first `fewer` items refill a plan that was never captured, with rows
    of another count: the smaller tiles a refill may choose fit as well."""
    text = f"2 {rows} {len(sizes)} {fewer} {more_rows}\n" + "\n".join(map(str, sizes)) + "\n"
    r = subprocess.run([str(refill_bin)], input=text, capture_output=True, text=True, check=True,
                       timeout=120)
    assert r.stdout.split("\n")[-2] == "allocs 0", r.stdout
