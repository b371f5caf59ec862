"""Radial operators on both sides of the line between the windowed pass's two kernels, which lies at
C G = 2048 grid points along y (register passes from there on, at G >= 128)."""

import numpy as np
import pytest
import torch

import workloads as w
from oracle import nufft, operator as op

pytestmark = pytest.mark.gpu
TOL = 1e-5  # the FP32 path's tolerance


def c64(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, dtype=np.complex64))).cuda()


@pytest.mark.parametrize("n,sigma,C", [
    (16, 2.0, 3), (32, 2.0, 33), (64, 1.5, 24), (64, 2.0, 15), (64, 2.0, 16), (96, 2.0, 10), (96, 2.0, 11),
    (128, 1.5, 11), (128, 2.0, 7), (128, 2.0, 8), (160, 2.0, 6), (160, 2.0, 7), (256, 2.0, 3), (256, 2.0, 4),
])
def test_windowed_pass_kernels(n, sigma, C):
    import paper_2008_09042_gb300 as mp

    q, rng = 3, np.random.default_rng(n + C)
    k = rng.uniform(-np.pi, np.pi, size=(300, 2)).astype(np.float32)
    U = w.smooth_orthonormal_basis(n, n, q, seed=1).astype(np.complex64).astype(np.complex128)
    a = w.random_coefficients(C, q, seed=2).astype(np.complex64).astype(np.complex128)
    p = w.random_image(n * n, seed=4).astype(np.complex64).astype(np.complex128)
    r = w.random_coefficients(C, len(k), seed=3, decay=False).astype(np.complex64).astype(np.complex128)
    ctx = mp.Context(0)
    plan = mp.Plan(ctx, (n, n), traj=k, kb_width=4, oversamp=sigma)
    B = mp.Basis(ctx, U.T)
    kb = nufft.KBGriddingNUFFT((n, n), k.astype(np.float64), W=4, sigma=sigma)
    for got, ref in ((mp.forward(ctx, plan, B, c64(a), c64(p)), op.forward(kb, U, a, p)),
                     (mp.adjoint(ctx, plan, B, c64(a), c64(r)), op.adjoint(kb, U, a, r))):
        assert np.linalg.norm(got.cpu().numpy() - ref) < TOL * np.linalg.norm(ref)
