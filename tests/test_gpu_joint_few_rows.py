"""The joint ALS row solvers on both sides of the rule between them (1,216 rows,
rank 28), with and without long rating rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 8, 15, 28, 29, 32])
@pytest.mark.parametrize("rows", [1, 7, 8, 9, 1216, 1217])
def test_rows_around_the_rule(R, rows):
    items, words = 700, 20
    g = torch.Generator().manual_seed(rows + R)
    counts = torch.randint(0, 6, (rows,), generator=g)
    counts[rows // 2] = 600  # one row of three pieces
    pairs = torch.cat([torch.stack([torch.full((int(n),), u), torch.randperm(items, generator=g)[:n]])
                       for u, n in enumerate(counts)], 1)
    yidx = pairs[:, torch.randperm(pairs.shape[1], generator=g)].to(torch.int32).contiguous()
    yval = 3 + torch.randn(yidx.shape[1], generator=g)
    dims = [rows, items, words]
    idx, val = synth.uniform_tensor(dims, min(5000, rows * 1000), seed=88, device="cuda")
    F = [f * 0.5 for f in synth.normal_factors(dims, R, seed=89, device="cuda")]
    mu, lam = 0.3, 0.5
    t = dfacto.Tensor(idx, val, dims, rank=R, lambda_reg=lam)
    t.set_factors(F)
    t.set_ratings(yidx.cuda(), yval.cuda(), mu)
    obj = t.joint_als_iter()
    ot, oy = oracle.Tensor(idx.cpu().numpy(), val.cpu().numpy(), dims), oracle.Ratings(yidx.numpy(), yval.numpy())
    st, Fo = oracle.joint_als_sweep(oy, ot, [f.double().cpu().numpy() for f in F], mu, lam)
    assert st == oracle.OK
    # FP32 Grams amplified by the solves, as in the stepwise test of the joint sweep
    for m, f in enumerate(t.factors()):
        assert np.linalg.norm(f.double().cpu().numpy() - Fo[m]) <= 1e-4 * np.linalg.norm(Fo[m]), m
    want = oracle.joint_loss(oy, ot, Fo, mu, lam)
    assert abs(obj - want) <= 1e-5 * abs(want)
