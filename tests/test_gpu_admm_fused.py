"""The fused image solver (maps kept for the solve) against the solve on the operator calls.

mpi_image_solve / mpi_image_solve_dynamic on 2D Cartesian plans run fused passes; with a fixed line
kernel they run on the operator calls instead.  Both are the same algorithm in FP32 with sums in
another order, so few iterations keep them within 1e-4 (a BF16 solve rounds the same basis and
coefficients on both routes, so the same bound holds).
"""

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def c64(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, dtype=np.complex64))).cuda()


def f64(t):
    return t.detach().cpu().numpy().astype(np.complex128)


def nrmse(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def mp():
    import paper_2008_09042_gb300 as mp

    return mp


def _mask(kind, ny, nx, seed):
    rng = np.random.default_rng(seed)
    m = np.zeros((ny, nx), dtype=bool)
    if kind == "lines":  # whole rows and empty ones
        m[rng.choice(ny, ny // 2, replace=False)] = True
    elif kind == "points":  # every row partly sampled
        m[:, ::3] = True
        m[::2, 1] = True
    elif kind == "mixed":  # whole, partial and empty rows
        m[: ny // 3] = True
        m[ny // 2, 5:9] = True
    elif kind == "one":
        m[ny // 2, nx // 2] = True
    return np.flatnonzero(m.ravel()).astype(np.int32)


@pytest.mark.parametrize("ny,nx,C,kind,frames,prec", [
    (64, 64, 4, "lines", 1, "fp32"),
    (16, 48, 1, "points", 1, "fp32"),
    (48, 16, 9, "mixed", 1, "fp32"),
    (320, 96, 3, "points", 1, "fp32"),
    (96, 320, 8, "lines", 1, "bf16"),
    (192, 128, 5, "mixed", 1, "mixed"),
    (32, 512, 2, "points", 1, "fp32_simt"),
    (512, 32, 2, "mixed", 1, "fp32"),
    (256, 64, 17, "points", 1, "mixed"),
    (128, 192, 3, "one", 1, "fp32"),
    (64, 48, 7, "points", 3, "fp32"),
    (48, 96, 2, "lines", 5, "bf16"),
])
def test_fused_solve_matches_the_operator_calls(mp, ny, nx, C, kind, frames, prec):
    q, N = 12, ny * nx
    U = w.smooth_orthonormal_basis(ny, nx, q, seed=3) * np.sqrt(N)
    idx = [_mask(kind, ny, nx, 5 + t) for t in range(frames)]
    M = len(idx[0])
    rng = np.random.default_rng(9)
    alpha = c64(w.random_coefficients(C, q, seed=4))
    y = c64(rng.normal(size=(frames, C, M)) + 1j * rng.normal(size=(frames, C, M)))
    eps = np.full((frames, C), 0.3 * np.sqrt(M))
    eps[0, 0] = 0.0  # a ball of radius zero
    out = []
    for line_kernel in (0, 8):
        ctx = mp.Context(0)
        ctx.set_line_kernel(line_kernel)
        B = mp.Basis(ctx, U.T)
        plans = [mp.Plan(ctx, (ny, nx), sample_idx=i) for i in idx]
        kw = dict(n_outer=4, n_cg=3, n_tv=11, prec=prec)
        if frames == 1:
            p, h = mp.image_solve(ctx, plans[0], B, alpha, y[0].contiguous(), eps[0], **kw)
        else:
            p, h = mp.image_solve_dynamic(ctx, plans, B, alpha, y, eps, **kw)
        ctx.synchronize()
        out.append((f64(p), h))
    assert nrmse(out[0][0], out[1][0]) < 1e-4
    np.testing.assert_allclose(out[0][1], out[1][1], rtol=1e-3)


def test_fused_solve_without_cg_steps(mp):
    # no CG step: the image stays zero and only the duals move
    ctx = mp.Context(0)
    plan = mp.Plan(ctx, (64, 64), sample_idx=_mask("points", 64, 64, 1))
    B = mp.Basis(ctx, w.smooth_orthonormal_basis(64, 64, 5, seed=1).T)
    y = torch.ones((2, plan.M), dtype=torch.complex64, device="cuda")
    p, h = mp.image_solve(ctx, plan, B, c64(w.random_coefficients(2, 5, seed=2)), y, np.ones(2), n_outer=3, n_cg=0,
                          n_tv=0)
    assert float(p.abs().max()) == 0.0 and np.isfinite(h).all()


@pytest.mark.parametrize("exponent", [-90, 90])
def test_fused_solve_of_data_whose_squares_leave_fp32(mp, exponent):
    # data and radii scaled by 2^e, rho by 2^-e: the image scales along; |y|^2 is 2^-180 or 2^180
    ny = nx = 64
    C, s = 3, 2.0 ** exponent
    idx = _mask("points", ny, nx, 1)
    U = w.smooth_orthonormal_basis(ny, nx, 8, seed=3) * np.sqrt(ny * nx)
    rng = np.random.default_rng(2)
    alpha = c64(w.random_coefficients(C, 8, seed=4))
    y = c64((rng.normal(size=(C, len(idx))) + 1j * rng.normal(size=(C, len(idx)))) * s)
    eps = np.full(C, 0.3 * np.sqrt(len(idx)) * s)
    out = []
    for line_kernel in (0, 8):
        ctx = mp.Context(0)
        ctx.set_line_kernel(line_kernel)
        p, h = mp.image_solve(ctx, mp.Plan(ctx, (ny, nx), sample_idx=idx), mp.Basis(ctx, U.T), alpha, y, eps,
                              n_outer=4, n_cg=3, n_tv=11, rho0=1.0 / s)
        ctx.synchronize()
        out.append((f64(p), h))
    assert float(np.linalg.norm(out[1][0])) > 0
    assert nrmse(out[0][0], out[1][0]) < 1e-4
    np.testing.assert_allclose(out[0][1], out[1][1], rtol=1e-3)
