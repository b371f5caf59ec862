"""A recorded batch after the context's workspace has grown: its kernels keep the block they were
recorded with."""

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def _slice(mp, ctx, n, C, q, seed, traj=False):
    rng = np.random.default_rng(seed)
    kw = dict(traj=rng.uniform(-np.pi, np.pi, size=(500, 2)).astype(np.float32)) if traj else \
        dict(sample_idx=np.flatnonzero(rng.random(n * n) < 0.3).astype(np.int32))
    plan = mp.Plan(ctx, (n, n), **kw)
    z = lambda *s: torch.from_numpy(w.random_image(s, seed=seed).astype(np.complex64)).cuda()  # noqa: E731
    return dict(plan=plan, basis=mp.Basis(ctx, w.random_image((q, n * n), seed=seed + 1).astype(np.complex64)),
                alpha=z(C, q), p=z(n * n), y=z(C, plan.M), x=z(n * n))


@pytest.mark.parametrize("traj", [False, True])
def test_batch_after_the_workspace_grew(traj):
    import paper_2008_09042_gb300 as mp

    ctx = mp.Context(0)
    a, b = _slice(mp, ctx, 64, 4, 6, 1, traj), _slice(mp, ctx, 96, 3, 5, 2, traj)
    batches = [mp.Batch(ctx, [a]), mp.Batch(ctx, [a, b])]
    batches[0].run()
    ctx.synchronize()
    want = a["y"].clone(), a["x"].clone()
    before = ctx.workspace_bytes()
    big = _slice(mp, ctx, 256, 24, 4, 3)
    mp.forward(ctx, big["plan"], big["basis"], big["alpha"], big["p"])
    assert ctx.workspace_bytes() > before
    other = torch.zeros(before, dtype=torch.uint8, device="cuda")  # may take the place of a freed block
    for i, batch in enumerate(batches * 2):
        a["y"].zero_(), a["x"].zero_()
        batch.run()
        ctx.synchronize()
        assert torch.equal(a["y"], want[0]) and torch.equal(a["x"], want[1])
        assert int(other.max()) == 0
        if i == 2:
            batches[0].close()
    third = mp.Batch(ctx, [b])
    third.run()
    ctx.synchronize()
    ctx.close()  # before its batches
    batches[1].close()
    third.close()
