"""The thermostat's variates of a whole segment are drawn before it, 8 steps to
a warp, beside its first factor: a segment and its steps one call after another
(one step of variates each) give the same bits, as long as the list of the first
step serves them all (the order of the kinetic energy's sum is the list's)."""
import numpy as np
import pytest

from paper_2005_08348_gb300 import mdas, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [2, 8, 9])
def test_a_segment_equals_its_steps(n, prec):
    m = synth.patch(128, 2, seed=51)
    whole, steps = (mdas.System(m, precision=prec) for _ in range(2))
    whole.md_steps(n, swap_every=0)
    for _ in range(n):
        steps.md_steps(1, swap_every=0)
    a, b = whole.get_state(), steps.get_state()
    for k in ("pos_u", "vel", "step"):
        assert np.array_equal(a[k], b[k]), k
    whole.close()
    steps.close()
