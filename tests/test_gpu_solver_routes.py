"""Which kernels a solve runs on: graphs recorded under another choice of FFT kernels are not replayed."""

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def _problem(mp, ctx, n=64, C=3, q=6):
    mask = np.zeros((n, n), dtype=bool)
    mask[::2] = True
    plan = mp.Plan(ctx, (n, n), sample_idx=np.flatnonzero(mask.ravel()).astype(np.int32))
    basis = mp.Basis(ctx, w.smooth_orthonormal_basis(n, n, q, seed=1).T * n)
    alpha = torch.from_numpy(w.random_coefficients(C, q, seed=2).astype(np.complex64)).cuda()
    y = torch.from_numpy(w.random_image((C, plan.M), seed=3).astype(np.complex64)).cuda()
    return plan, basis, alpha, y, np.full(C, 0.1 * np.sqrt(plan.M))


def _solve(mp, ctx, problem):
    """Kernels of a solve whose graph has been recorded (recording it may launch some too), and the image."""
    plan, basis, alpha, y, eps = problem
    for _ in range(2):
        n0 = ctx.launches()
        p, _ = mp.image_solve(ctx, plan, basis, alpha, y, eps, n_outer=3, n_cg=2, n_tv=4)
        ctx.synchronize()
    return ctx.launches() - n0, p


def test_line_kernel_choice_between_solves():
    import paper_2008_09042_gb300 as mp

    want = {}
    for choice in (0, 8):
        ctx = mp.Context(0)
        ctx.set_line_kernel(choice)
        want[choice] = _solve(mp, ctx, _problem(mp, ctx))
    assert want[0][0] != want[8][0]  # the fused passes and the operator calls
    ctx = mp.Context(0)
    problem = _problem(mp, ctx)
    for choice in (0, 8, 0, 8):
        ctx.set_line_kernel(choice)
        n, p = _solve(mp, ctx, problem)
        assert n == want[choice][0]
        assert torch.equal(p, want[choice][1])


def test_solve_returns_to_the_fused_route_after_a_failed_allocation():
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    fused, _ = _solve(mp, ctx, _problem(mp, ctx))
    ctx.set_line_kernel(8)
    calls, _ = _solve(mp, ctx, _problem(mp, ctx))  # both routes' kernels are loaded
    ctx.set_line_kernel(0)
    # 64 coils of 512^2: 268 MB of maps and coil images on the fused route, 50 MB on the operator calls
    n, C = 512, 64
    mask = np.zeros((n, n), dtype=bool)
    mask[::64] = True
    plan = mp.Plan(ctx, (n, n), sample_idx=np.flatnonzero(mask.ravel()).astype(np.int32))
    basis = mp.Basis(ctx, w.smooth_orthonormal_basis(n, n, 4, seed=1).T * n)
    alpha = torch.from_numpy(w.random_coefficients(C, 4, seed=2).astype(np.complex64)).cuda()
    y = torch.from_numpy(w.random_image((C, plan.M), seed=3).astype(np.complex64)).cuda()
    problem = plan, basis, alpha, y, np.full(C, 0.1 * np.sqrt(plan.M))
    ctx.reserve(plan, basis, C)
    mp.forward(ctx, plan, basis, alpha, torch.zeros(n * n, dtype=torch.complex64, device="cuda"))
    ctx.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (150 << 20), dtype=torch.uint8, device="cuda")
    n0, p0 = _solve(mp, ctx, problem)
    assert n0 >= calls
    del fill
    torch.cuda.empty_cache()
    n1, p1 = _solve(mp, ctx, problem)
    assert n1 <= fused
    a, b = p0.cpu().numpy(), p1.cpu().numpy()
    assert np.linalg.norm(a - b) < 1e-4 * np.linalg.norm(a)  # the routes' bound (test_gpu_admm_fused.py)


@pytest.mark.parametrize("choice", [-2, -3])
def test_choices_for_volumes_leave_2d_calls_alone(choice):
    import paper_2008_09042_gb300 as mp

    def counts(c):
        ctx = mp.Context(0)
        ctx.set_line_kernel(c)
        problem = _problem(mp, ctx)
        n, p = _solve(mp, ctx, problem)
        plan, basis, alpha, y, _ = problem
        slices = [dict(plan=plan, basis=basis, alpha=alpha, p=p, y=y.clone(), x=torch.empty_like(p)) for _ in range(5)]
        batch = mp.Batch(ctx, slices)
        return n, batch.kernels()

    assert counts(choice) == counts(0)
