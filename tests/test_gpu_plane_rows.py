"""The plane passes' choice of rows along y, over all nine plane shapes.

The planes of the volume have no row with samples, one, two in one residue class (mod NY/8, the inverse's
first step, or mod 8, the forward's second), whole and partial rows, and many rows.  Against the FP64 oracle at the FP32 operators' tolerance (1e-5).
"""

import numpy as np
import pytest
import torch

import workloads as w
from oracle import fourier, operator as op, tucker

pytestmark = pytest.mark.gpu


def c64(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, dtype=np.complex64))).cuda()


def rel(t, ref):
    x = t.cpu().numpy().astype(np.complex128)
    return float(np.linalg.norm(x - ref) / np.linalg.norm(ref))


def _mask(nz, ny, nx):
    rng = np.random.default_rng(ny + nx)
    rows = [[], [0], [ny - 1], [3, 3 + ny // 8], [5, 13], [ny // 2, ny // 2 + 1, 7], list(range(0, ny, 8)),
            list(range(ny // 8)), sorted(rng.choice(ny, 35, replace=False)), list(range(1, 34))]
    m = np.zeros((nz, ny, nx), dtype=bool)
    for z in range(nz):
        for k, y in enumerate(rows[z % len(rows)]):
            m[z, y] = True if (k + z) % 3 else rng.random(nx) < 0.4
            m[z, y, nx // 2] = True
    return m


@pytest.mark.parametrize("ny", [64, 96, 128])
@pytest.mark.parametrize("nx", [64, 96, 128])
def test_plane_rows(ny, nx):
    import paper_2008_09042_gb300 as mp

    dims, ranks, q, C = (32, ny, nx), (6, 8, 8), 9, 7
    ctx = mp.Context(0)
    core, fac = w.smooth_tucker_basis(dims, ranks, q, seed=27)
    core = core.astype(np.complex64).astype(np.complex128)
    fac = [f.astype(np.complex64).astype(np.complex128) for f in fac]
    tb = tucker.TuckerBasis(core, fac)
    idx = np.flatnonzero(_mask(*dims).ravel()).astype(np.int32)
    Fs = fourier.CartesianSampling(dims, idx)
    a = w.random_coefficients(C, q, seed=29).astype(np.complex64).astype(np.complex128)
    p = w.random_image(int(np.prod(dims)), seed=30).astype(np.complex64).astype(np.complex128)
    r = w.random_coefficients(C, idx.size, seed=31, decay=False).astype(np.complex64).astype(np.complex128)
    plan, B = mp.Plan(ctx, dims, sample_idx=idx), mp.TuckerBasis(ctx, core, fac)
    ctx.profile(True)
    assert rel(mp.forward(ctx, plan, B, c64(a), c64(p)), op.forward(Fs, tb, a, p)) < 1e-5
    assert rel(mp.adjoint(ctx, plan, B, c64(a), c64(r)), op.adjoint(Fs, tb, a, r)) < 1e-5
    ctx.synchronize()
    _, kern = ctx.profile_read(kernels=True)
    assert {"k_plane_pipe<fwd>", "k_plane_pipe<inv>"} <= set(kern)
