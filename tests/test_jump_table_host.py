"""The MWC jump table between streams, on the CPU: the library's table code over
stand-ins for the CUDA runtime's calls (native/jump_table_check.cu).  A call on
another stream than the table's waits for the build, also where that stream has the
handle of one that was destroyed; a rebuild waits for the device while calls of
other streams may read the table."""
from __future__ import annotations

import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]


@pytest.fixture(scope="module")
def table_bin(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not Path(nvcc).exists():
        pytest.skip("nvcc not found")
    out = tmp_path_factory.mktemp("table") / "jump_table_check"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                    "-I", str(ROOT / "include"), "-I", str(ROOT / "paper_1101_1846_gb300" / "csrc"),
                    "-o", str(out), str(ROOT / "tests" / "native" / "jump_table_check.cu")],
                   check=True, capture_output=True, timeout=600)
    return out


# calls (handle, id, rows, segs, ready) and what each gets (table, events, syncs)
BUILD = ((64, 1, 64, 8, 0), (1, 0, 1))  # the first one allocates
CASES = {
    "one stream": [BUILD, ((64, 1, 64, 8, 0), (1, 0, 0)), ((64, 1, 64, 4, 1), (1, 0, 0)),
                   ((64, 1, 32, 8, 0), (1, 0, 0)), ((64, 1, 64, 8, 1), (0, 0, 0))],
    "another stream": [BUILD, ((128, 2, 64, 8, 0), (1, 1, 0)), ((64, 1, 32, 8, 0), (1, 0, 1))],
    "a destroyed stream's handle, read": [BUILD, ((64, 2, 64, 8, 0), (1, 1, 0)),
                                          ((64, 2, 64, 8, 1), (1, 1, 0))],
    "a destroyed stream's handle, rebuilt": [BUILD, ((64, 2, 32, 8, 0), (1, 0, 1)),
                                             ((64, 2, 64, 8, 0), (1, 0, 0))],
    "no table after four waits": [BUILD, *[((64, 2 + i, 32 << i % 2, 8, 0), (1, 0, 1))
                                           for i in range(4)], ((64, 7, 32, 8, 0), (0, 0, 0)),
                                  ((64, 7, 64, 16, 0), (1, 0, 1))],
}


@pytest.mark.parametrize("name", CASES)
def test_table_waits_for_other_streams(table_bin, name):
    calls, want = zip(*CASES[name])
    r = subprocess.run([str(table_bin)], input="\n".join(" ".join(map(str, c)) for c in calls),
                       capture_output=True, text=True, check=True, timeout=120)
    assert [tuple(map(int, x.split())) for x in r.stdout.strip().split("\n")] == list(want)
