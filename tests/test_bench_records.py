"""bench.py reads the grouped expansions' figures from the library's tuning records."""

import numpy as np
import pytest

import bench


def test_figures_of_a_record():
    rec = ("grouped expansion (16 slices, N=102400, q=160, sumC=288, fp32): 152 CTAs, bundles of 0, skew 0: 296.10 us;"
           " 152 CTAs, bundles of 32, skew 0: 223.04 us; chose 152, bundles of 32, skew 0 (223.04 us)")
    g = bench.grouped_expansion(rec, 6692.1, 1950.9)
    assert (g["slices"], g["N"], g["q"], g["coils"], g["ctas"], g["bundle_coils"]) == (16, 102400, 160, 288, 152, 32)
    assert g["us_per_launch"] == 223.04
    assert g["tflops"] == pytest.approx(2 * 102400 * 320 * 576 / 223.04e-6 / 1e12)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_every_record_of_a_batch_has_figures(prec):
    import torch

    import paper_2008_09042_gb300 as mp
    import workloads as w

    ctx = mp.Context(0)
    n, q = 64, 8
    basis = mp.Basis(ctx, w.smooth_orthonormal_basis(n, n, q, seed=1).T)
    plan = mp.Plan(ctx, (n, n), sample_idx=np.arange(0, n * n, 3, dtype=np.int32))
    z = lambda *s: torch.zeros(s, dtype=torch.complex64, device="cuda")  # noqa: E731
    slices = [dict(plan=plan, basis=basis, alpha=z(C, q), p=z(n * n), y=z(C, plan.M), x=z(n * n)) for C in (2, 9, 4)]
    batch = mp.Batch(ctx, slices, kind="pair", prec=prec)
    recs = [r for r in ctx.tuning_records() if r.startswith("grouped expansion")]
    assert len(recs) == 1
    g = bench.grouped_expansion(recs[0], 6692.1, 1950.9)
    assert (g["slices"], g["N"], g["q"], g["coils"]) == (3, n * n, q, 15) and g["us_per_launch"] > 0
    batch.close()
