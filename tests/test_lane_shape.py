"""The CTA shape of waves that overlap on lanes (laned.lane_shape), on the CPU:
lists on both sides of the line, whose tiles are counted as the library does."""
from __future__ import annotations

import pytest

pytest.importorskip("torch")

from paper_1101_1846_gb300.laned import LANE_TILES, lane_shape  # noqa: E402
from paper_1101_1846_gb300.scheduler import Piece  # noqa: E402

SMS = 152


@pytest.mark.parametrize("sizes,over", [
    ([1], False), ([512] * LANE_TILES * SMS, False), ([512] * LANE_TILES * SMS + [1], True),
    ([513] * (LANE_TILES * SMS // 2), False), ([513] * (LANE_TILES * SMS // 2 + 1), True),
    ([512 * LANE_TILES * SMS], False), ([65_536] * 20, True), ([32] * 1000, True)])
def test_shape_of_overlapping_waves(sizes, over):
    wave = [Piece(i, 0, 1024) for i in range(len(sizes))]
    assert lane_shape(wave, sizes, 2, SMS) == ((512, 1) if over else (0, 0))
    assert lane_shape(wave, sizes, 1, SMS) == (0, 0)
