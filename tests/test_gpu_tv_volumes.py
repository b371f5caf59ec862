"""mpi_tv_prox on both sides of the line between the fused 3D iteration and the one that forms x
first (64 MB of dual variables), against the oracle's FP64 iterations; and its use of the
context's workspace."""

import numpy as np
import pytest
import torch

import workloads as w
from oracle import solvers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(96, 96, 96), (64, 128, 128), (128, 96, 96)])
@pytest.mark.parametrize("n_iter", [0, 1, 3])
def test_tv_prox_of_large_volumes(dims, n_iter):
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    plan = mp.Plan(ctx, dims, sample_idx=np.arange(4, dtype=np.int32))
    v = w.random_image(int(np.prod(dims)), seed=7).astype(np.complex64)
    x = mp.tv_prox(ctx, plan, torch.from_numpy(v).cuda(), 0.15, n_iter).cpu().numpy()
    ref = solvers.tv_prox(v.astype(np.complex128), 0.15, dims, n_iter)
    assert np.linalg.norm(x - ref) < 1e-5 * np.linalg.norm(ref)  # as for the other TV tests


def test_tv_prox_between_solves():
    # the prox grows the workspace that the recorded solve's kernels use
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    n, C, q = 64, 2, 4
    plan = mp.Plan(ctx, (n, n), sample_idx=np.arange(0, n * n, 3, dtype=np.int32))
    basis = mp.Basis(ctx, w.smooth_orthonormal_basis(n, n, q, seed=1).T)
    y = torch.from_numpy(w.random_image((C, plan.M), seed=2).astype(np.complex64)).cuda()
    first = mp.sm_estimate(ctx, plan, basis, y, C, n_outer=2, n_cg=3)
    before = ctx.workspace_bytes()
    big = mp.Plan(ctx, (64, 64, 128), sample_idx=np.arange(4, dtype=np.int32))
    v = torch.from_numpy(w.random_image(64 * 64 * 128, seed=3).astype(np.complex64)).cuda()
    x = mp.tv_prox(ctx, big, v, 0.2, 4)
    assert ctx.workspace_bytes() > before
    again = mp.sm_estimate(ctx, plan, basis, y, C, n_outer=2, n_cg=3)
    assert torch.equal(first[0], again[0]) and torch.equal(first[1], again[1])
    assert torch.equal(x, mp.tv_prox(ctx, big, v, 0.2, 4))
