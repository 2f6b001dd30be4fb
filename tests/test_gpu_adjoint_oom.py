"""An adjoint call whose scratch does not fit returns what it took, and can be tried again.

The allocator hook refuses the fourth allocation of the call (host-side; nothing is
launched on what there is), twice, and then serves them all.
"""
import pytest

pytestmark = pytest.mark.gpu


def test_failed_adjoint_allocation_takes_no_memory():
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
    own = capi._alloc_cbs
    assert lib.ifdlbm_set_allocator(hooks[0], hooks[1], None) == 0
    try:
        s = Solver([cavity(33, 29, 400.0, 0.75)], kernel="staged", dt_mode="grid")
    finally:
        assert lib.ifdlbm_set_allocator(own[0], own[1], None) == 0
    s.step(3)
    state = torch.zeros(capi.ifdlbm_state_bytes(s.h) // 8, dtype=torch.float64, device="cuda")
    adj, dp = torch.zeros_like(state), torch.zeros(3, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    capi.ifdlbm_save_state_dev(s.h, state)
    before = s.info(0).device_bytes
    for _ in range(2):
        left[0] = 3
        with pytest.raises(capi.IfdlbmError) as e:
            capi.ifdlbm_adjoint_seed_energy(s.h, state, adj, dp)
        assert e.value.code == capi.IFDLBM_ERR_OOM
        assert s.info(0).device_bytes == before
    left[0] = 10 ** 9
    capi.ifdlbm_adjoint_seed_energy(s.h, state, adj, dp)
    s.sync()
    assert s.info(0).device_bytes > before and float(adj.abs().max()) > 0
    s.close()
