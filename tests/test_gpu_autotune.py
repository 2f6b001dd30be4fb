"""The autotuner offers the layouts that the handle's own rules give.

A 65^2 cavity runs with 2 rows a task; 16 or more leave most of the chip idle (three
times the time). And the layout a handle runs is itself a candidate, so that what is
kept is no slower: one that is in none of the lists is timed besides them.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_small_cavity_keeps_few_rows():
    from paper_2306_07603_gb300.solver import Solver, cavity
    s, ref = (Solver([cavity(65, 65, 100.0, 0.75)], precision="fp32dev") for _ in range(2))
    t = s.autotune(trial_steps=50)
    assert t.fused_rows < 16 and t.schedule in (0, 1), (t.fused_rows, t.schedule)
    assert s.info(0).ntasks == t.ntasks
    for h in (s, ref):
        h.step(7)
    f, g = (h.get_state(0)[0] for h in (s, ref))
    assert np.abs(f - g).max() <= 1e-6 * np.abs(f).max()
    s.close()
    ref.close()


def test_present_layout_is_a_candidate():
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(129, 97, 100.0, 0.75)], precision="fp32dev", fused_threads=128, fused_rows=37)
    assert s.autotune(trial_steps=2).candidates == 46
    s.close()
