"""Radial adjoints whose samples crowd into few grid cells: the spreading then gives every warp and
thread one group of four coils, whatever the coil count and the grid would allow."""

import numpy as np
import pytest
import torch

import workloads as w
from oracle import nufft, operator as op

pytestmark = pytest.mark.gpu
TOL = 1e-5  # the FP32 path's tolerance


def c64(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, dtype=np.complex64))).cuda()


@pytest.mark.parametrize("n,W,C,M,power", [
    (256, 4, 12, 6000, 4.0),  # one group: the fullest cell holds most of the samples
    (256, 3, 12, 6000, 0.0),  # three groups
    (256, 2, 20, 3000, 0.5),  # three groups with padded coils
    (160, 2, 12, 4000, 3.0),
    (32, 6, 17, 5000, 1.0),   # every cell dense
    (32, 8, 1, 1, 0.0),
])
def test_crowded_cells(n, W, C, M, power):
    import paper_2008_09042_gb300 as mp

    q, rng = 3, np.random.default_rng(n + W)
    k = (rng.uniform(-np.pi, np.pi, size=(M, 2)) * rng.random((M, 1)) ** power).astype(np.float32)
    U = w.smooth_orthonormal_basis(n, n, q, seed=1).astype(np.complex64).astype(np.complex128)
    a = w.random_coefficients(C, q, seed=2).astype(np.complex64).astype(np.complex128)
    r = w.random_coefficients(C, M, seed=3, decay=False).astype(np.complex64).astype(np.complex128)
    ctx = mp.Context(0)
    plan = mp.Plan(ctx, (n, n), traj=k, kb_width=W, oversamp=2.0)
    x = mp.adjoint(ctx, plan, mp.Basis(ctx, U.T), c64(a), c64(r)).cpu().numpy()
    ref = op.adjoint(nufft.KBGriddingNUFFT((n, n), k.astype(np.float64), W=W, sigma=2.0), U, a, r)
    assert np.linalg.norm(x - ref) < TOL * np.linalg.norm(ref)
