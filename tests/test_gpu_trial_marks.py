"""An exchange trial that runs beside the next MD step marks the step items it can
change; only those sum their forces again after an accepted exchange.  Marks of
trials before the call must not be there any more, however the trial counter has
gone on since (the bitmap of a trial is that of its counter's parity): the items
counted after other trials in between are those of a system that never marked any
(separate launches give the same states and do not mark)."""
import numpy as np
import pytest

from paper_2005_08348_gb300 import mdas, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("between", ["exchange", "speculative", "mutation", "restore"])
def test_marks_of_earlier_trials_do_not_last(between):
    accepted = 0
    for seed in (1, 2, 3, 4):
        m = synth.patch(700, 3, seed=seed)
        runs = [mdas.System(m, temperature=3000.0) for _ in range(2)]
        runs[1].set_persistent(False)
        redos = []
        for s in runs:
            s.md_steps(12, swap_every=5)                 # trials 0 and 1, marked beside steps 6 and 11
            s.set_persistent(True)
            if between == "exchange":
                s.swap_trials(1)
            elif between == "speculative":
                s.set_trial_path("speculative")
                s.swap_trials(1)
            elif between == "mutation":
                s.mutation_trials(1)
            else:
                st = s.get_state()
                st["trial"] += 1
                s.resume(st)
            before = s.counters()["item_redos"]
            s.md_steps(9, swap_every=4)                  # trial 3 beside step 5, trial 4 beside step 9
            redos.append(s.counters()["item_redos"] - before)
        a, b = (s.get_state() for s in runs)
        for k in ("pos_u", "vel", "ltype"):
            assert np.array_equal(a[k], b[k]), k
        assert redos[0] == redos[1]
        accepted += int(runs[0].trial_log(3, 1)[0]["accepted"])
        for s in runs:
            s.close()
    assert accepted > 0                                  # (a rejected trial has no item sum again)
