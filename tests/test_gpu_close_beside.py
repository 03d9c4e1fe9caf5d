"""The close of a step (thermostat factor, kinetic energy) beside the next
step's items, where a lone system is too large for the overlapped mode and in
the share of a batch: the bits of the separate kernels and of the system alone,
with and without a trial after the step, over list builds."""
import numpy as np
import pytest

from paper_2005_08348_gb300 import mdas, synth

pytestmark = pytest.mark.gpu


def _same(a, b):
    x, y = a.get_state(), b.get_state()
    for k in ("pos_u", "vel", "ltype", "step", "trial"):
        assert np.array_equal(x[k], y[k]), k
    assert a.counters()["accepted"] == b.counters()["accepted"]


# 1700 lipids: 1339 items for the 1216 groups of 152 blocks
@pytest.mark.parametrize("prec,lanes,every,calls", [
    ("fp32", 4, 0, (1, 2, 12)), ("fp32", 2, 1, (7,)), ("fp32", 4, 3, (1, 8, 6)), ("fp64", 4, 2, (1, 6))])
def test_lone_system_beyond_the_overlapped_mode(prec, lanes, every, calls):
    m = synth.patch(1700, 3, seed=71)
    runs = [mdas.System(m, precision=prec, list_skin=0.15) for _ in range(2)]
    runs[1].set_persistent(False)
    for s in runs:
        s.set_list_lanes(lanes)
        for n in calls:
            s.md_steps(n, swap_every=every)
    assert runs[0].counters()["list_builds"] >= 2
    _same(*runs)
    for s in runs:
        s.close()


def test_lambda_blocks_of_a_large_system():
    m = synth.patch(1700, 3, seed=72)
    runs = [mdas.System(m) for _ in range(2)]
    runs[1].set_persistent(False)
    res = [s.alchemical_move(4, 5, 3) for s in runs]
    # 40 work terms (8 lipids, 5 blocks) of fewer than 2500 pairs below 10^4
    # kJ/mol, some 40 rounded FP64 operations each: 40 * 1.1e-7 kJ/mol
    assert abs(res[0]["w"] - res[1]["w"]) < 5e-6 and res[0]["accepted"] == res[1]["accepted"]
    _same(*runs)
    for s in runs:
        s.close()


@pytest.mark.parametrize("sizes", [(128, 142), (700, 128, 300), (1152, 200, 200, 900)])
def test_shares_of_a_batch(sizes):
    ms = [synth.patch(n, 2 + k % 2, seed=73 + k, system_id=k) for k, n in enumerate(sizes)]
    batch, alone = ([mdas.System(m, list_skin=0.2) for m in ms] for _ in range(2))
    for n in (1, 14):
        mdas.batch_run(batch, n, 5)
        for s in alone:
            s.md_steps(n, swap_every=0)
            s.swap_trials(5)
    for b, a in zip(batch, alone):
        _same(b, a)
    for s in batch + alone:
        s.close()
