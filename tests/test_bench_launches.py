"""The kernel count the benchmark reports for its timed region."""

import pytest


@pytest.mark.parametrize("steps,bodies,want", [(20, 2, 22), (16, 1, 17), (17, 1, 19), (200, 2, 213), (20, 0, 20), (1, 1, 2)])
def test_step_launches(steps, bodies, want):
    """One step kernel per step; with bodies, one sum of the loads for every 16 steps begun."""
    import bench

    assert bench.step_launches(steps, bodies) == want
