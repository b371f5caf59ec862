"""The fused image solver over the magnitudes of the maps.

The sums of the CG grow as the fourth power of the maps and shrink with their square, so they leave
FP32's range long before the vectors do.  The solve on the operator calls (a fixed line kernel) has
the same vectors in FP32 and FP64 sums.  Both are the same algorithm with the same FP32 roundings per
step in another order, so a few iterations keep them within 1e-4, as for maps of magnitude one.
"""

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def c64(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, dtype=np.complex64))).cuda()


@pytest.mark.parametrize("scale_basis", [False, True])
@pytest.mark.parametrize("exponent", [-70, -34, 0, 32])
def test_fused_solve_of_maps_whose_sums_leave_fp32(exponent, scale_basis):
    import paper_2008_09042_gb300 as mp

    ny = nx = 64
    C, q, s = 3, 8, 2.0 ** exponent
    m = np.zeros((ny, nx), dtype=bool)
    m[:, ::3] = True
    m[::2, 1] = True
    idx = np.flatnonzero(m.ravel()).astype(np.int32)
    U = w.smooth_orthonormal_basis(ny, nx, q, seed=3) * np.sqrt(ny * nx)
    rng = np.random.default_rng(2)
    alpha = w.random_coefficients(C, q, seed=4)
    y = c64(rng.normal(size=(C, idx.size)) + 1j * rng.normal(size=(C, idx.size)))
    eps = np.full(C, 0.3 * np.sqrt(idx.size))
    if scale_basis:
        U = U * s
    else:
        alpha = alpha * s
    out = []
    for line_kernel in (0, 8):
        ctx = mp.Context(0)
        ctx.set_line_kernel(line_kernel)
        p, h = mp.image_solve(ctx, mp.Plan(ctx, (ny, nx), sample_idx=idx), mp.Basis(ctx, U.T), c64(alpha), y, eps,
                              n_outer=4, n_cg=3, n_tv=11)
        ctx.synchronize()
        out.append((p.cpu().numpy().astype(np.complex128), h))
    (a, ha), (b, hb) = out
    assert np.isfinite(a).all() and np.linalg.norm(b) > 0
    assert np.linalg.norm(a - b) < 1e-4 * np.linalg.norm(b)
    np.testing.assert_allclose(ha, hb, rtol=1e-3)
