"""What the inputs of the GPU tests of trials and moves exercise, by the oracle:
trials that an earlier acceptance of their chunk reaches (they must be evaluated
again), and moves of either outcome."""
import numpy as np
import pytest

import oracle
from paper_2005_08348_gb300 import synth

RC = 1.1


def _reached(m, o, pos_u, records, chunk, lipid_of):
    """Trials after an accepted one of their chunk that draw one of its lipids or
    a lipid with a bead within rc of it (by the records' chunks of this length)."""
    bpl = m.lipid_bead_type.shape[1]
    box = np.asarray(m.box)
    pos = pos_u[: len(m.lipid_type) * bpl].astype(np.float64).reshape(-1, bpl, 3) / 2.0 ** 32 * box

    def near(a, b):
        d = pos[a][:, None] - pos[b][None]
        d -= box * np.round(d / box)
        return a == b or (d * d).sum(-1).min() < RC * RC

    n = 0
    for c in range(0, len(records), chunk):
        part = records[c:c + chunk]
        for k, r in enumerate(part):
            n += not r["null"] and any(e["accepted"] and any(near(x, y) for x in lipid_of(e) for y in lipid_of(r))
                                       for e in part[:k])
    return n


# the calls of test_gpu_trial_chain.py's exchange test (without its largest system)
@pytest.mark.parametrize("lipids,types,chunk,n", [(700, 3, 43, 130), (700, 2, 43, 87), (200, 3, 256, 300)])
def test_exchange_chains_meet(lipids, types, chunk, n):
    m = synth.patch(lipids, types, seed=31)
    o = oracle.Oracle(m, temperature=500.0)
    st = o.state()
    _, rec = o.swap_trials(st["pos_u"], st["ltype"], 0, n)
    assert _reached(m, o, st["pos_u"], rec, chunk, lambda r: (r["a"], r["b"])) >= 3


@pytest.mark.parametrize("lipids,types,chunk,n", [(300, 3, 18, 18), (700, 2, 43, 44), (200, 3, 256, 40)])
def test_mutation_chains_meet(lipids, types, chunk, n):
    m = synth.patch(lipids, types, seed=32)
    o = oracle.Oracle(m, temperature=500.0)
    st = o.state()
    rec, _ = o.mutation_trials(st["pos_u"], st["ltype"], 0, n, [0.0, 0.7, -0.4][:types])
    assert sum(r["accepted"] for r in rec) > 0
    assert _reached(m, o, st["pos_u"], rec, chunk, lambda r: (r["a"],)) >= 1


def test_batched_chains_meet():
    reached = 0
    for k, n in enumerate((128, 700, 300)):
        m = synth.patch(n, 2 + k % 2, seed=40 + k, system_id=k)
        o = oracle.Oracle(m)
        st = o.state()
        _, rec = o.swap_trials(st["pos_u"], st["ltype"], 0, 100)
        reached += _reached(m, o, st["pos_u"], rec, 43, lambda r: (r["a"], r["b"]))
    assert reached >= 3


def test_moves_have_both_outcomes():
    """The moves of test_gpu_move_pairs.py: accepted ones for every pair count, and
    rejected ones."""
    rejected = 0
    for lipids, types, n_pairs in ((128, 2, 1), (128, 2, 64), (300, 3, 33), (700, 3, 64)):
        m = synth.patch(lipids, types, seed=61)
        o = oracle.Oracle(m, temperature=3000.0)
        st = o.state()
        outcomes = []
        for _ in range(4):
            outcomes.append(o.mdas_move(st, n_pairs, 1, 0)["accepted"])   # (st takes the move)
        assert True in outcomes, (lipids, n_pairs)
        rejected += outcomes.count(False)
    assert rejected > 0
