"""The N-body step's weight 1 / (x * sqrt(x)) against the rounded operations,
for every float the step evaluates it for."""
import pytest

pytestmark = pytest.mark.gpu


def test_weight_is_the_rounded_operations():
    from paper_2503_10516_gb300 import igs
    assert igs.selftest_nbody_weight() == 0
