"""The orbital dipole in pointing periods of few nodes, where one thread takes a period (up to 24 nodes):
either side of that line, more periods than a block's threads, beside longer ones.  Oracle and bound of
test_gpu_orbital_short_periods.py."""
import pytest

from tests.test_gpu_orbital_short_periods import test_short_periods as check

pytestmark = pytest.mark.gpu
TINY = tuple(range(27))


@pytest.mark.parametrize("nodes", [(23, 24, 25, 26), TINY * 12, (24,) * 127 + (25, 300, 2), TINY + (257, 0, 24, 3000)])
@pytest.mark.parametrize("s", [2, 7])
def test_tiny_periods(nodes, s):
    check(nodes, s)
