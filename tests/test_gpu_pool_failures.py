"""A member's failed allocation in lbve_pool_residuals leaves the pool as it was: no snapshot
is taken, the pool goes on, and a later call gives what a first call gives."""
import numpy as np
import pytest

from gpu_helpers import require_gpu
from test_gpu_pool import _members

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


# the residual's buffers are two allocations: the velocity snapshot and the block sums
@pytest.mark.parametrize("refused", ["first", "second"])
def test_residuals_out_of_memory(refused):
    import torch

    from paper_2009_12279_gb300 import LbveError, Solver, lbve, serve

    reqs = _members("f32")
    stream = torch.cuda.Stream()
    pool = lbve.Pool("f32", budget_bytes=10**10, stream=stream.cuda_stream)
    held, refusing = {}, []

    def alloc(nbytes, st):
        if refusing and refusing.pop(0):
            return 0
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(ptr, nbytes, st):
        torch.cuda.synchronize()
        held.pop(ptr)

    solvers = []
    for k, r in enumerate(reqs):
        s = serve.build_solver(r, "f32", stream.cuda_stream)
        if k == 2:  # the same solve on caller-provided memory
            p = s.params
            s.close()
            s = Solver(params=p, stream=stream.cuda_stream, allocator=(alloc, free))
            s.set_geometry(r.flags, r.wall_vel)
            if r.particle is not None:
                q = r.particle
                s.add_particle(q["X"], q["R"], q["rho_p"], Fext=q["Fext"])
        pool.admit(s)
        solvers.append(s)
    pool.step(60)
    refusing[:] = [True] if refused == "first" else [False, True]
    with pytest.raises(LbveError, match="LBVE_ENOMEM"):
        pool.residuals()
    refusing.clear()
    pool.step(40)
    got = pool.residuals()
    for r, s, (res, norm) in zip(reqs, solvers, got):
        assert norm > 0.0 and res == 1.0, r.kind  # against a zero snapshot
    pool.step(100)
    again = pool.residuals()
    for r, s, (res, norm) in zip(reqs, solvers, again):
        alone = serve.build_solver(r, "f32", stream.cuda_stream)
        alone.step(100)
        assert alone.residual()[0] == 1.0
        alone.step(100)
        assert alone.residual() == (res, norm), r.kind
        assert np.array_equal(alone.read_pdfs(), s.read_pdfs())
        alone.close()
    pool.close()
