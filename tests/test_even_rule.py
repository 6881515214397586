"""The rule that evens out a plain call's CTAs (even_threads in
csrc/gen_kernels.cuh), evaluated on the CPU: at most whole waves, and where they
would be exactly whole the last streams' CTA has a place of its own unless the
CTAs cannot be widened for it."""
from __future__ import annotations

import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]
SMS = 152
MWC, XOR128, KISS, XORSHIFT8 = 0, 1, 2, 4


@pytest.fixture(scope="module")
def even_bin(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not Path(nvcc).exists():
        pytest.skip("nvcc not found")
    out = tmp_path_factory.mktemp("even") / "even_check"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                    "-I", str(ROOT / "include"), "-I", str(ROOT / "paper_1101_1846_gb300" / "csrc"),
                    "-o", str(out), str(ROOT / "tests" / "native" / "even_check.cu")],
                   check=True, capture_output=True, timeout=600)
    return out


def per_cta(threads, realigned):
    return 31 * (threads // 32) + 1 if realigned else threads


@pytest.mark.parametrize("kind,fmt", [(MWC, 0), (MWC, 1), (XOR128, 0), (XOR128, 1), (KISS, 0),
                                      (KISS, 1), (XORSHIFT8, 0)])
@pytest.mark.parametrize("realigned", [0, 1])
def test_waves(even_bin, kind, fmt, realigned):
    most = 512 if kind == XORSHIFT8 else 128 if kind == XOR128 and not realigned else 256
    groups = list(range(19_500, 460_000, 7)) + [340_345 // 4, 226_649 // 4, 378_017 // 4]
    fixed = per_cta(512, realigned)
    text = "".join(f"{kind} {fmt} {g} {fixed} {1 - realigned} {realigned} {realigned}\n"
                   for g in groups)
    r = subprocess.run([str(even_bin)], input=text, capture_output=True, text=True, check=True,
                       timeout=120)
    chosen = list(map(int, r.stdout.split()))
    assert len(chosen) == len(groups) and any(chosen)
    alone = kind != XORSHIFT8 and not (realigned and fmt == 1 and kind != MWC)
    for g, t in zip(groups, chosen):
        if t == 0:
            continue
        assert t % 32 == 0 and 32 <= t <= most
        ctas = -(-g // per_cta(t, realigned))
        waves = -(-ctas // SMS)
        if ctas < SMS * waves or not realigned:
            continue
        # exactly whole waves and the last streams' CTA after them
        wider = t + 32
        assert wider > most or -(-wider // 128) > -(-t // 128) or (waves > 2 and not alone), g
