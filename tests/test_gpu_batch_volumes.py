"""Batches of volumes on a dense basis: every slice's values are those of its own calls, bit for bit,
also where a group is large enough for the 2D slices' grouped FFT passes and where slices of one basis
have grids of equal size and row length that are split differently into planes and rows."""

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu

A, B_, C_ = (16, 32, 48), (32, 16, 48), (512, 48)


@pytest.mark.parametrize("grids,groups", [
    ([A] * 3, 1),
    ([A] * 5, 1),  # enough slices for grouped passes
    ([A, A, B_, B_, C_, C_], 3),
    ([A] * 4 + [C_] * 4 + [B_] * 4, 3),
    ([A, C_, B_, A], 0),
])
@pytest.mark.parametrize("kind,prec", [("pair", "fp32"), ("pair", "bf16"), ("adjoint", "fp32")])
def test_batched_volumes_match_single_calls(grids, groups, kind, prec):
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    N, q = int(np.prod(A)), 6
    rng = np.random.default_rng(1)
    U = (rng.normal(size=(q, N)) + 1j * rng.normal(size=(q, N))).astype(np.complex64)
    basis = mp.Basis(ctx, U)
    slices = []
    for i, dims in enumerate(grids):
        C = 1 + 3 * i % 7
        idx = np.flatnonzero(rng.random(N) < 0.2).astype(np.int32)
        y = (rng.normal(size=(C, idx.size)) + 1j * rng.normal(size=(C, idx.size))).astype(np.complex64)
        slices.append(dict(plan=mp.Plan(ctx, dims, sample_idx=idx), basis=basis, y=torch.from_numpy(y).cuda(),
                           alpha=torch.from_numpy(w.random_coefficients(C, q, seed=i).astype(np.complex64)).cuda(),
                           p=torch.from_numpy(w.random_image(N, seed=i).astype(np.complex64)).cuda(),
                           x=torch.zeros(N, dtype=torch.complex64, device="cuda")))
    batch = mp.Batch(ctx, slices, kind=kind, prec=prec)
    assert batch.groups() == groups
    batch.run()
    ctx.synchronize()
    for s in slices:
        y1 = s["y"] if kind == "adjoint" else mp.forward(ctx, s["plan"], basis, s["alpha"], s["p"], prec)
        assert torch.equal(s["y"], y1)
        assert torch.equal(s["x"], mp.adjoint(ctx, s["plan"], basis, s["alpha"], y1, prec))
    batch.close()
