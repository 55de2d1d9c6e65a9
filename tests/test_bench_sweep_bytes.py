"""The bytes per site-update that the bench counts for its whole-grid sweep:
48 a level, half of that where the call takes levels in pairs."""
import pytest

import bench


@pytest.mark.parametrize("side, steps, scratch, want", [
    (128, 256, 8, 48.0),              # one level per pass
    (1280, 128, 24, 24.0), (512, 64, 24, 24.0),
    (512, 6, 24, 48.0 * (1 - 0.5 * 4 / 6)),  # four levels in pairs, two by themselves
    (512, 3, 24, 48.0),
])
def test_sweep_bytes_follow_the_passes(side, steps, scratch, want):
    sites = side ** 3
    assert bench.sweep_bytes_per_update(sites, steps, scratch * sites) == pytest.approx(want)
