"""The TV prox written over its own input."""

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(320, 192), (16, 32, 48)])
@pytest.mark.parametrize("lam,n_iter", [(0.0, 3), (0.3, 0), (0.3, 1), (0.3, 10), (0.3, 23)])
def test_tv_prox_in_place(dims, lam, n_iter):
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    N = int(np.prod(dims))
    plan = mp.Plan(ctx, dims, sample_idx=np.arange(5, dtype=np.int32))
    v = torch.from_numpy(w.random_image(N, seed=1).astype(np.complex64)).cuda()
    want = mp.tv_prox(ctx, plan, v, lam, n_iter)
    x = v.clone()
    assert ctx.lib.mpi_tv_prox(ctx.h, plan.h, x.data_ptr(), lam, n_iter, x.data_ptr()) == 0
    assert torch.equal(x, want)
