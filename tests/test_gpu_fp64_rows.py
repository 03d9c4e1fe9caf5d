"""The FP64 step keeps the entries that may be inside rc as bits, 64 rows of a
bead's list at a time: lists of a few rows, and of 64 and more in one column.

As for the step kernel's forces elsewhere: from rest and without a thermostat
one step gives v = F dt / m, so F = v m / dt is compared with the oracle's at
1e-10 of max(|F_i|, F_rms), the FP64 force tolerance."""
import numpy as np
import pytest

import oracle
from _systems import beads
from paper_2005_08348_gb300 import mdas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,lanes", [(5, 4), (9, 4), (9, 2), (12, 4), (12, 2)])
def test_lists_of_any_length_match_oracle(side, lanes):
    rng = np.random.default_rng(side)
    g = (np.stack(np.meshgrid(*[np.arange(side)] * 3), -1).reshape(-1, 3) + 0.5) * (4.0 / side)
    m = beads(g + rng.uniform(-0.02, 0.02, g.shape), rng.integers(0, 10, side ** 3))
    m.dt = 0.002
    s = mdas.System(m, precision="fp64", tau_t=0.0)
    s.set_list_lanes(lanes)
    st = s.get_state()
    s.md_steps(1, swap_every=0)
    F = s.get_state()["vel"] * (m.mass / m.dt)
    _, Fo = oracle.Oracle(m).energy(st["pos_u"])
    frms = np.sqrt((Fo * Fo).sum(1).mean())
    err = np.linalg.norm(F - Fo, axis=1) / np.maximum(np.linalg.norm(Fo, axis=1), frms)
    assert err.max() < 1e-10, err.max()
    s.close()
