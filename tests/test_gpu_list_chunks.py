"""The list build fetches its candidates 32 at a time, two chunks ahead: a box of
three list cells along every edge, so that every bead is a candidate, with fewer
beads than a chunk, whole chunks, and one more or less.

From rest and without a thermostat one step gives v = F dt / m: F = v m / dt at
1e-5 (FP32) and 1e-10 (FP64) of max(|F_i|, F_rms), the step kernel's force
tolerances."""
import numpy as np
import pytest

import oracle
from _systems import beads
from paper_2005_08348_gb300 import mdas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 96, 97])
def test_few_candidates_match_oracle(n, prec):
    rng = np.random.default_rng(n)
    pts = [np.array([0.1, 0.1, 3.9]), np.array([3.9, 0.1, 0.3])]     # a pair across the box's faces
    while len(pts) < n:
        p = rng.uniform(0.0, 4.0, 3)
        d = np.asarray(pts) - p
        d -= 4.0 * np.round(d / 4.0)
        if (d * d).sum(1).min() > 0.4 ** 2:
            pts.append(p)
    m = beads(pts, rng.integers(0, 10, n))
    m.dt = 0.002
    s = mdas.System(m, precision=prec, tau_t=0.0)
    st = s.get_state()
    s.md_steps(1, swap_every=0)
    F = s.get_state()["vel"] * (m.mass / m.dt)
    _, Fo = oracle.Oracle(m).energy(st["pos_u"])
    frms = np.sqrt((Fo * Fo).sum(1).mean())
    err = np.linalg.norm(F - Fo, axis=1) / np.maximum(np.linalg.norm(Fo, axis=1), frms)
    assert err.max() < (1e-10 if prec == "fp64" else 1e-5), err.max()
    s.close()
