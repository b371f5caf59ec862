"""Batches whose groups are large enough for grouped FFT passes (all coils of a group's slices in one
launch): every slice's values are those of its own calls, bit for bit, whatever mix of masks, coil
counts and tuned kernels the group holds."""

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def _idx(kind, ny, nx, i):
    m = np.zeros((ny, nx), dtype=bool)
    if kind == "lines":
        m[i % 3::3] = True
    elif kind == "points":
        m[:, i % 2::5] = True
    elif kind == "corner":
        m[ny - 1, nx - 2:] = True
    return np.flatnonzero(m.ravel()).astype(np.int32)


@pytest.mark.parametrize("ny,nx,kinds,coils", [
    (64, 64, ("points",), (1, 3, 8, 16, 32)),
    (128, 48, ("lines", "points", "empty"), (4, 9, 4, 9, 2, 24)),
    (256, 256, ("points", "lines"), (8, 16, 32, 8)),
    (48, 320, ("corner", "points"), (5, 6, 7, 8)),
    (320, 96, ("lines",), (2, 12, 3, 1)),
])
@pytest.mark.parametrize("kind,prec", [("pair", "fp32"), ("pair", "bf16"), ("forward", "fp32"), ("adjoint", "fp32")])
def test_grouped_passes_match_single_calls(ny, nx, kinds, coils, kind, prec):
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    q = 8
    B = mp.Basis(ctx, w.smooth_orthonormal_basis(ny, nx, q, seed=1).T)
    rng = np.random.default_rng(3)
    slices = []
    for i, C in enumerate(coils):
        idx = _idx(kinds[i % len(kinds)], ny, nx, i)
        plan = mp.Plan(ctx, (ny, nx), sample_idx=idx)
        y = (rng.normal(size=(C, idx.size)) + 1j * rng.normal(size=(C, idx.size))).astype(np.complex64)
        slices.append(dict(plan=plan, basis=B, y=torch.from_numpy(y).cuda(),
                           alpha=torch.from_numpy(w.random_coefficients(C, q, seed=i).astype(np.complex64)).cuda(),
                           p=torch.from_numpy(w.random_image(ny * nx, seed=i).astype(np.complex64)).cuda(),
                           x=torch.zeros(ny * nx, dtype=torch.complex64, device="cuda")))
    batch = mp.Batch(ctx, slices, kind=kind, prec=prec)
    assert batch.groups() == 1
    # grouped: an expansion, at most one pass along y per kernel and one row pass per direction
    assert batch.kernels() < (4 * len(slices) + 2) // (1 if kind == "pair" else 2)
    for _ in range(2):
        batch.run()
    ctx.synchronize()
    for s in slices:
        y1 = s["y"] if kind == "adjoint" else mp.forward(ctx, s["plan"], B, s["alpha"], s["p"], prec)
        assert torch.equal(s["y"], y1)
        if kind != "forward":
            assert torch.equal(s["x"], mp.adjoint(ctx, s["plan"], B, s["alpha"], y1, prec))
    batch.close()


@pytest.mark.parametrize("n,q,coils", [
    (320, 160, (32, 8, 16, 1, 32)),  # the largest coefficient operand (a ring of two stages) beside small ones
    (16, 5, (1, 3, 2)),              # fewer tiles than CTAs
    (32, 30, tuple(1 + i % 7 for i in range(170))),  # more slices than SMs
])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_grouped_expansions_of_mixed_coil_counts(n, q, coils, prec):
    # every CTA lays out its own slice's operand, accumulators and ring: values as in the slice's own calls
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    B = mp.Basis(ctx, w.smooth_orthonormal_basis(n, n, q, seed=1).T)
    slices = []
    for i, C in enumerate(coils):
        idx = _idx("points", n, n, i)
        slices.append(dict(plan=mp.Plan(ctx, (n, n), sample_idx=idx), basis=B,
                           y=torch.zeros((C, idx.size), dtype=torch.complex64, device="cuda"),
                           alpha=torch.from_numpy(w.random_coefficients(C, q, seed=i).astype(np.complex64)).cuda(),
                           p=torch.from_numpy(w.random_image(n * n, seed=i).astype(np.complex64)).cuda(),
                           x=torch.zeros(n * n, dtype=torch.complex64, device="cuda")))
    batch = mp.Batch(ctx, slices, kind="pair", prec=prec)
    assert batch.groups() == 1
    batch.run()
    ctx.synchronize()
    for s in slices:
        y1 = mp.forward(ctx, s["plan"], B, s["alpha"], s["p"], prec)
        assert torch.equal(s["y"], y1)
        assert torch.equal(s["x"], mp.adjoint(ctx, s["plan"], B, s["alpha"], y1, prec))
    batch.close()
