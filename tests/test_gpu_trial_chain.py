"""Trials in order, many per launch (k_chain_*): exchanges over the pair lists
and mutations over the cells against the oracle's one-after-another processing,
at the edges of a chunk (n_lip / 16 trials, none evaluated ahead below 16, 256
at most) and over several calls, whose chunks and type updates must not leak
into the next (exchanges read the list-ordered types, mutations the cells').

dE sums fewer than 2500 pair terms below 10^4 kJ/mol in FP64, some 40 rounded
operations each: 2500 * 10^4 * 40 * 2^-53 = 1.1e-7 kJ/mol, taken as 1e-6."""
import math

import numpy as np
import pytest

import oracle
from paper_2005_08348_gb300 import mdas, synth

pytestmark = pytest.mark.gpu
TOL = 1e-6


def _check(rec, want, shift, kT):
    for g, r in zip(rec, want):
        assert (g["a"], g["b"], bool(g["null"]), g["u"]) == (r["a"], r["b"], bool(r["null"]), r["u"])
        if r["null"]:
            assert g["dE"] == 0.0 and not g["accepted"]
            continue
        assert abs(g["dE"] - r["dE"]) < TOL
        if abs(r["dE"] - shift(r) + kT * math.log(r["u"])) > TOL:
            assert bool(g["accepted"]) == bool(r["accepted"])


# chunks of 43 (700 lipids), 18 (300), 256 (4200); 200 lipids: chunks of 12 would be too short
@pytest.mark.parametrize("lipids,types,lanes,calls", [
    (700, 3, 4, (1, 15, 16, 43, 44, 130)), (700, 2, 2, (87, 2)), (200, 3, 2, (300, 17)), (4200, 3, 4, (257,))])
def test_exchanges_in_order_match_oracle(lipids, types, lanes, calls):
    m = synth.patch(lipids, types, seed=31)
    s = mdas.System(m, temperature=500.0)
    s.set_list_lanes(lanes)
    o = oracle.Oracle(m, temperature=500.0)
    st = s.get_state()
    lt, t0 = st["ltype"], 0
    for n in calls:
        stats, rec = s.swap_trials(n)
        lt, want = o.swap_trials(st["pos_u"], lt, t0, n)
        _check(rec, want, lambda r: 0.0, o.kT)
        assert np.array_equal(s.get_state()["ltype"], lt)
        assert stats["accepted"] == sum(r["accepted"] for r in want)
        t0 += n
    assert s.counters()["accepted"] > 0
    s.close()


@pytest.mark.parametrize("lipids,types,calls", [(300, 3, (18, 19)), (700, 2, (44, 1)), (200, 3, (40,))])
def test_mutations_in_order_match_oracle(lipids, types, calls):
    m = synth.patch(lipids, types, seed=32)
    s = mdas.System(m, temperature=500.0)
    o = oracle.Oracle(m, temperature=500.0)
    mu = [0.0, 0.7, -0.4][:types]
    st = s.get_state()
    lt, t0 = st["ltype"], 0
    for n in calls:
        _, rec = s.mutation_trials(n, mu=mu)
        want, after = o.mutation_trials(st["pos_u"], lt, t0, n, mu)
        cur = np.array(lt)
        for g, r in zip(rec, want):
            _check([g], [r], lambda r: mu[r["b"]] - mu[cur[r["a"]]], o.kT)
            if r["accepted"]:
                cur[r["a"]] = r["b"]
        assert np.array_equal(s.get_state()["ltype"], after)
        lt, t0 = after, t0 + n
        # the exchanges that follow read the list-ordered types
        _, rec = s.swap_trials(20)
        lt, want = o.swap_trials(st["pos_u"], lt, t0, 20)
        _check(rec, want, lambda r: 0.0, o.kT)
        t0 += 20
    s.close()


def test_chains_of_a_batch_equal_the_systems_alone():
    """The largest system sets a batch's chunks; the records do not depend on them."""
    ms = [synth.patch(n, 2 + k % 2, seed=40 + k, system_id=k) for k, n in enumerate((128, 700, 300))]
    batch, alone = ([mdas.System(m) for m in ms] for _ in range(2))
    mdas.batch_run(batch, 0, 100)
    for b, a in zip(batch, alone):
        _, rec = a.swap_trials(100)
        assert b.trial_log(0, 100).tobytes() == rec.tobytes()
        assert np.array_equal(a.get_state()["ltype"], b.get_state()["ltype"])
    for x in batch + alone:
        x.close()
