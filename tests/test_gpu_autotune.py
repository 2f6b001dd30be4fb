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


def test_a_trial_that_does_not_fit_leaves_state_and_layout():
    """The allocator hook refuses the tables of a finer layout: the call fails, the handle is as
    it was and steps on as one that was never tuned."""
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    left = [10 ** 9]

    def alloc(nbytes, stream, ctx):
        left[0] -= 1
        return torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0)) if left[0] >= 0 else None

    def free(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    hooks = capi.ALLOC_FN(alloc), capi.FREE_FN(free)
    lib = capi.load_library()
    capi.use_torch_allocator()
    assert lib.ifdlbm_set_allocator(hooks[0], hooks[1], None) == 0
    try:
        s = Solver([cavity(129, 97, 100.0, 0.75)], precision="fp32dev", fused_rows=64)
    finally:
        assert lib.ifdlbm_set_allocator(capi._alloc_cbs[0], capi._alloc_cbs[1], None) == 0
    ref = Solver([cavity(129, 97, 100.0, 0.75)], precision="fp32dev", fused_rows=64)
    for h in (s, ref):
        h.step(5)
    before = s.info(0)
    left[0] = 1                                        # the saved state, and no more
    with pytest.raises(capi.IfdlbmError) as e:
        s.autotune(trial_steps=2)
    assert e.value.code == capi.IFDLBM_ERR_OOM and "fused layout" in str(e.value)
    left[0] = 10 ** 9
    after = s.info(0)
    assert (after.fused_rows, after.ntasks, after.device_bytes) == (64, before.ntasks, before.device_bytes)
    for h in (s, ref):
        h.step(3)
    assert np.array_equal(s.get_state(0)[0], ref.get_state(0)[0])
    t = s.autotune(trial_steps=2)
    assert t.candidates == 45 and s.info(0).ntasks == t.ntasks
    s.close()
    ref.close()
