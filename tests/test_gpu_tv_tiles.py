"""mpi_tv_prox against the oracle at the edges of its tiles and launches (2D: tiles with their halo
in shared memory, up to ten iterations per launch; 3D: a launch per iteration).  FP32 against FP64,
1e-5 as for the other TV tests."""

import numpy as np
import pytest
import torch

import workloads as w
from oracle import solvers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(16, 16), (32, 48), (48, 320), (512, 96), (16, 32, 64), (48, 16, 96)])
@pytest.mark.parametrize("n_iter", [0, 1, 9, 10, 11, 21])
def test_tv_prox_tiles_and_launches(dims, n_iter):
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    plan = mp.Plan(ctx, dims, sample_idx=np.arange(4, dtype=np.int32))
    v = w.random_image(int(np.prod(dims)), seed=7).astype(np.complex64).astype(np.complex128)
    vg = torch.from_numpy(v.astype(np.complex64)).cuda()
    x = mp.tv_prox(ctx, plan, vg, 0.15, n_iter).cpu().numpy().astype(np.complex128)
    ref = solvers.tv_prox(v, 0.15, dims, n_iter)
    assert np.linalg.norm(x - ref) / np.linalg.norm(ref) < 1e-5
