"""Plans of their own on several host threads: a launch of one thread is not refused because another
thread launches the same kernel with less shared memory. Every plan here has levels above 48 KB per
CTA, of different sizes, in the same kernel instances."""
import threading

import numpy as np
import pytest
import torch

import paper_1809_10573_gb300 as P
from paper_1809_10573_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("mode,fmt,dt,R,adjoint", [
    (P.MODE_FP64, P.STORE_C128, torch.complex128, 7, False), (P.MODE_FP64, P.STORE_C128, torch.complex128, 7, True),
    (P.MODE_DF64, P.STORE_DF64, torch.complex128, 1, False), (P.MODE_TF32X3, P.STORE_C64, torch.complex64, 32, False)])
def test_applies_of_several_threads_do_not_refuse_each_other(mode, fmt, dt, R, adjoint):
    jobs = []
    for leaf, N in ((64, 1 << 13), (128, 1 << 12), (256, 1 << 13)):
        plan = P.Plan.build(*inputs.uniform_grid(N), eps=1e-8, leaf=leaf, kernel="fio", sign=-1, rank_cap=120)
        plan.set_storage(fmt)
        plan.reserve(R)
        if R == 1:
            plan.set_level_variants(mode, [1] * (plan.L + 1))   # a streaming kernel on every level
        xs = torch.from_numpy(inputs.complex_gaussian(N, R, seed=N)).cuda().to(dt).t().contiguous().t()
        ref, ys = torch.empty_like(xs), torch.empty_like(xs)
        plan.apply_raw(xs.data_ptr(), ref.data_ptr(), R, N, mode, 0, adjoint)
        jobs.append((plan, xs, ref, ys, torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(len(jobs))

    def work(plan, xs, ref, ys, stream):
        try:
            start.wait()
            for _ in range(300):
                plan.apply_raw(xs.data_ptr(), ys.data_ptr(), R, plan.N, mode, stream.cuda_stream, adjoint)
        except Exception as e:  # a refused launch
            errors.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for plan, xs, ref, ys, _ in jobs:
        assert torch.equal(ref, ys)
