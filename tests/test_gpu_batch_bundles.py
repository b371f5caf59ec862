"""Grouped FP32 expansions whose slices are bundled (several slices' coefficients in one operand):
every slice's values are those of its own calls, bit for bit, forward and adjoint.  Most slices have
few coils, so that streaming the basis once per bundle instead of once per slice is a third of the
work and the timed choice between the layouts is not in doubt; the tuning record says which ran."""

import re

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("big", [(9, 17), (32,), (8, 16, 24)])
def test_bundled_slices_match_single_calls(big):
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    n, q = 128, 96
    rng = np.random.default_rng(1)
    U = (rng.normal(size=(q, n * n)) + 1j * rng.normal(size=(q, n * n))).astype(np.complex64)
    basis = mp.Basis(ctx, U)
    idx = np.flatnonzero(rng.random(n * n) < 0.25).astype(np.int32)
    plan = mp.Plan(ctx, (n, n), sample_idx=idx)
    coils = [1, 5, 3, 8, 2, 7] * 4
    for i, C in enumerate(big):
        coils.insert(5 * i + 2, C)
    slices = [dict(plan=plan, basis=basis, y=torch.zeros((C, plan.M), dtype=torch.complex64, device="cuda"),
                   alpha=torch.from_numpy(w.random_coefficients(C, q, seed=i).astype(np.complex64)).cuda(),
                   p=torch.from_numpy(w.random_image(n * n, seed=i).astype(np.complex64)).cuda(),
                   x=torch.zeros(n * n, dtype=torch.complex64, device="cuda")) for i, C in enumerate(coils)]
    batch = mp.Batch(ctx, slices, kind="pair", prec="fp32")
    rec = [r for r in ctx.tuning_records() if r.startswith("grouped expansion")]
    assert len(rec) == 1 and int(re.search(r"chose \d+, bundles of (\d+)", rec[0]).group(1)) > 0, rec
    batch.run()
    ctx.synchronize()
    for s in slices:
        y = mp.forward(ctx, plan, basis, s["alpha"], s["p"])
        assert torch.equal(s["y"], y)
        assert torch.equal(s["x"], mp.adjoint(ctx, plan, basis, s["alpha"], y))
    batch.close()
