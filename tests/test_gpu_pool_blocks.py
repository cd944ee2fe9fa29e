"""Pool calls of more steps than one replayed graph holds: bitwise the solves stepped alone,
wall forces, particles and rounding keys included, whatever the lengths of the calls."""
import numpy as np
import pytest

from gpu_helpers import require_gpu
from test_gpu_pool import _members, _state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _requests(precision, copies):
    return [r for _ in range(copies) for r in _members(precision)]


# 4 members (all with kernels of their own, some 14 kernels a step: blocks of up to 290 steps) and
# 68 (small ones in the batched kernels)
@pytest.mark.parametrize("precision,copies,calls", [("bf16", 1, (1, 300, 300)), ("f32", 1, (601,)),
                                                    ("bf16", 17, (161, 160)), ("f64", 1, (330, 331))])
def test_long_calls_equal_alone(precision, copies, calls):
    import torch

    from paper_2009_12279_gb300 import lbve, serve

    reqs = _requests(precision, copies)
    stream = torch.cuda.Stream()
    pool = lbve.Pool(precision, budget_bytes=10**11, stream=stream.cuda_stream)
    solvers = [serve.build_solver(r, precision, stream.cuda_stream) for r in reqs]
    for s in solvers:
        pool.admit(s)
    for n in calls:
        pool.step(n)
    refs = []
    for r in reqs[:4]:
        s = serve.build_solver(r, precision, stream.cuda_stream)
        s.step(sum(calls))
        refs.append((_state(s), s.read_particle(0) if r.particle else None, s.body_forces()))
        s.close()
    for k, s in enumerate(solvers):
        ref, pref, bref = refs[k % 4]
        assert s.time == sum(calls)
        for a, b in zip(_state(s), ref):
            assert np.array_equal(a, b), f"member {k} ({reqs[k].kind})"
        if pref is not None:
            p = s.read_particle(0)
            assert all(np.array_equal(p[q], pref[q]) for q in ("X", "v", "w"))
        assert np.array_equal(s.body_forces(), bref)
    pool.close()
