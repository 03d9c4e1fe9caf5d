"""kernel_launches counts what a mutation call launches: three kernels per chunk
of trials evaluated ahead (n_lip / 16 trials, from 16 trials on), one per 256
trials otherwise."""
import pytest

from paper_2005_08348_gb300 import mdas, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lipids,trials,launches", [
    (300, 15, 1), (300, 16, 3), (300, 18, 3), (300, 19, 6), (200, 256, 1), (200, 300, 2)])
def test_mutations_count_their_launches(lipids, trials, launches):
    s = mdas.System(synth.patch(lipids, 3, seed=5))
    before = s.counters()["kernel_launches"]
    s.mutation_trials(trials, log=False)
    assert s.counters()["kernel_launches"] - before == launches
    s.close()
