"""List-build tasks of 1, 2, 4 or 8 beads, by the beads there are for the grid's
warps (4864 with 152 blocks): the lists, and so the bits, of the separate
kernels, whose tasks have 8."""
import numpy as np
import pytest

from paper_2005_08348_gb300 import mdas, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [4, 2])
@pytest.mark.parametrize("lipids", [128, 192, 194, 368, 372, 768, 770])
def test_lists_do_not_depend_on_the_tasks(lipids, lanes):
    m = synth.patch(lipids, 3, seed=91)
    runs = [mdas.System(m, list_skin=0.1) for _ in range(2)]
    runs[1].set_persistent(False)
    for s in runs:
        s.set_list_lanes(lanes)
        s.md_steps(12, swap_every=4)
    assert runs[0].counters()["list_builds"] >= 3
    a, b = (s.get_state() for s in runs)
    for k in ("pos_u", "vel", "ltype"):
        assert np.array_equal(a[k], b[k]), k
    for s in runs:
        s.close()
