"""Contexts on two host threads are independent: launches that need different amounts of dynamic
shared memory of the same kernels (a limit that belongs to the kernel, not to a context) do not
disturb each other."""

import threading

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def _tv(mp, ctx, size):
    n, n_iter = ((256, 10), (64, 1))[size]
    plan = mp.Plan(ctx, (n, n), sample_idx=np.arange(n, dtype=np.int32))
    v = torch.from_numpy(w.random_image(n * n, seed=size).astype(np.complex64)).cuda()
    return lambda: mp.tv_prox(ctx, plan, v, 0.1, n_iter)


def _simt(mp, ctx, size):
    n, q, C = ((32, 200, 48), (32, 8, 2))[size]
    plan = mp.Plan(ctx, (n, n), sample_idx=np.arange(n * n, dtype=np.int32))
    basis = mp.Basis(ctx, w.random_image((q, n * n), seed=1).astype(np.complex64))
    a = torch.from_numpy(w.random_coefficients(C, q, seed=2).astype(np.complex64)).cuda()
    p = torch.from_numpy(w.random_image(n * n, seed=3).astype(np.complex64)).cuda()
    r = torch.from_numpy(w.random_image((C, plan.M), seed=4).astype(np.complex64)).cuda()
    return lambda: torch.cat([t.flatten() for t in mp.jacobian_adjoint(ctx, plan, basis, a, p, r, "fp32_simt")])


@pytest.mark.parametrize("make", [_tv, _simt])
def test_shared_memory_limits_of_two_threads(make):
    import paper_2008_09042_gb300 as mp

    errors = []
    start = threading.Barrier(2)

    def work(size):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                ctx = mp.Context(0, stream)
                call = make(mp, ctx, size)
                want = call()
                stream.synchronize()
                start.wait(60)
                for _ in range(400):
                    got = call()
                stream.synchronize()
                assert torch.equal(got, want)
                ctx.synchronize()
        except Exception as e:  # reported by the test's thread
            start.abort()
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
