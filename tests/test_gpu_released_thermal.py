"""Fluctuating solvents against the values of an earlier release (released_values.py)."""
import pytest

import released_values as rv

pytestmark = pytest.mark.gpu


# As for the chains: 2e-5 of the array's norm is what single-precision results may differ by.  Noise that
# differs in its last bits stays far below that in FP32 (2e-7 of the velocities) and goes beyond it once it
# is rounded to 16 bits or moves stiff beads.
@pytest.mark.parametrize("name", sorted(rv.CASES["thermal"]))
def test_thermal_as_released(name):
    want, got = rv.golden("thermal"), rv.run("thermal", name)
    for key, value in got.items():
        d = rv.distance(value, want[name + "." + key])
        assert d <= 2e-5, (key, d)
