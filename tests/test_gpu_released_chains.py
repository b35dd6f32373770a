"""Chains against the values of an earlier release (released_values.py)."""
import pytest

import released_values as rv

pytestmark = pytest.mark.gpu


# The same arithmetic gives the same bits.  Allowed is what single-precision results may differ by from
# one release to the next: 2e-5 of the array's norm.  A last bit of the constraint solve or of a reciprocal
# that is rounded differently goes beyond it in these cases.
@pytest.mark.parametrize("name", sorted(rv.CASES["chain"]))
def test_chain_as_released(name):
    want, got = rv.golden("chain"), rv.run("chain", name)
    for key, value in got.items():
        d = rv.distance(value, want[name + "." + key])
        assert d <= 2e-5, (key, d)
