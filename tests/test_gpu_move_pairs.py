"""Pair selection draws 32 candidates at a time and marks and accepts with 128
threads: one pair, the 64 that a move may have (128 lipids), and fewer lipids
than they would take, whose candidates run out."""
import numpy as np
import pytest

import oracle
from paper_2005_08348_gb300 import mdas, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaflets", [False, True])
@pytest.mark.parametrize("lipids,types,n_pairs", [(128, 2, 1), (128, 2, 64), (300, 3, 33), (700, 3, 64)])
def test_pairs_marks_and_acceptance_match_oracle(lipids, types, n_pairs, leaflets):
    m = synth.patch(lipids, types, seed=61)
    s = mdas.System(m, temperature=3000.0)
    o = oracle.Oracle(m, temperature=3000.0)
    outcomes = set()
    for move in range(4):
        st = s.get_state()
        lt = st["ltype"]
        if leaflets:
            want = o.interleaflet_pairs(st["pos_u"], lt, move, n_pairs)
            res = s.interleaflet_move(n_pairs, 1, 0)
        else:
            want = o.mdas_pairs(lt, move, n_pairs)
            res = s.alchemical_move(n_pairs, 1, 0)
        assert np.array_equal(np.asarray(res["pairs"]).reshape(-1, 2), want)
        after = lt.copy()
        if res["accepted"]:
            after[want[:, 0]], after[want[:, 1]] = lt[want[:, 1]], lt[want[:, 0]]
        assert np.array_equal(s.get_state()["ltype"], after)
        # the beads' types are the lipids' again: energies of the new types
        e, _ = o.energy(st["pos_u"], ltype=after, forces=False)
        assert abs(s.energy()["potential"] - e["total"]) <= 1e-9 * abs(e["total"])
        outcomes.add(bool(res["accepted"]))
    s.close()
