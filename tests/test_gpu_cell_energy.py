"""The energy pass takes a cell's beads and its candidates 32 at a time and each
pair once, with the neighbour cells ahead: cells of 2 to 64 beads (one chunk of
32, one more than it, two), three cells or more along an edge.

Each term sums n pair terms of about 15 rounded operations in FP64, some of
them large and of either sign: 1e-9 of the sum of the magnitudes, bounded from
below by |LJ| + |RF| of the oracle, leaves a thousand times that for n = 1e5."""
import numpy as np
import pytest

import oracle
from _systems import beads
from paper_2005_08348_gb300 import mdas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("side", [4, 9, 10, 12])
@pytest.mark.parametrize("box", [(4.0, 4.0, 4.0), (4.0, 5.6, 4.7)])
def test_cells_of_any_occupancy_match_oracle(side, box, prec):
    rng = np.random.default_rng(side)
    g = (np.stack(np.meshgrid(*[np.arange(side)] * 3), -1).reshape(-1, 3) + 0.5) / side
    pts = g * np.asarray(box) + rng.uniform(-0.05, 0.05, (side ** 3, 3))
    m = beads(pts, rng.integers(0, 10, side ** 3), box=box)
    s = mdas.System(m, precision=prec)
    e = s.energy()
    want, _ = oracle.Oracle(m).energy(s.get_state()["pos_u"], forces=False)
    assert e["pairs"] == want["pairs"] > 0
    for k in ("lj", "rf"):
        assert abs(e[k] - want[k]) <= 1e-9 * (abs(want["lj"]) + abs(want["rf"])), k
    s.close()
