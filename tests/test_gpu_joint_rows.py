"""Joint ALS rows with more ratings than one piece (256): rows at and around
that length and its multiples, starting on and off a piece boundary, next to empty rows, for both
sides and ranks that fill and do not fill the row solver's layouts."""
import numpy as np
import pytest
import torch

import oracle
from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [dfacto.F32, dfacto.BF16])
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("R", [1, 5, 8, 12, 16, 24, 32])
def test_long_rating_rows(R, swap, dtype):
    counts = [1024, 1025, 0, 2500, 7, 0, 1, 3071, 40, 256, 257, 255] + [3] * 40
    users, items, words = len(counts), 3100, 20
    g = torch.Generator().manual_seed(77 + R)
    pairs = torch.cat([torch.stack([torch.full((n,), u), torch.randperm(items, generator=g)[:n]])
                       for u, n in enumerate(counts)], 1)
    pairs = pairs[:, torch.randperm(pairs.shape[1], generator=g)]
    dims = [users, items, words]
    if swap:
        pairs, dims = pairs.flip(0), [items, users, words]
    yidx = pairs.to(torch.int32).contiguous()
    yval = 3 + torch.randn(yidx.shape[1], generator=g)
    idx, val = synth.uniform_tensor(dims, 5000, seed=88, device="cuda")
    F = [f * 0.5 for f in synth.normal_factors(dims, R, seed=89, device="cuda")]
    mu, lam = 0.3, 0.5
    t = dfacto.Tensor(idx, val, dims, rank=R, lambda_reg=lam, factor_dtype=dtype)
    t.set_factors(F)
    t.set_ratings(yidx.cuda(), yval.cuda(), mu)
    before = [f.double().cpu().numpy() for f in t.factors()]
    obj = t.joint_als_iter()
    ot = oracle.Tensor(idx.cpu().numpy(), val.cpu().numpy(), dims)
    oy = oracle.Ratings(yidx.numpy(), yval.numpy())
    st, Fo = oracle.joint_als_sweep(oy, ot, before, mu, lam)
    assert st == oracle.OK
    got = [f.double().cpu().numpy() for f in t.factors()]
    if dtype == dfacto.BF16:
        # each side starts from the stored (rounded) factors: the oracle's B from
        # the GPU's A is the first update of the problem with users and items
        # exchanged; C has no ratings
        oys = oracle.Ratings(yidx.flip(0).contiguous().numpy(), yval.numpy())
        ots = oracle.Tensor(idx[[1, 0, 2]].contiguous().cpu().numpy(), val.cpu().numpy(),
                            [dims[1], dims[0], dims[2]])
        st, Fs = oracle.joint_als_sweep(oys, ots, [before[1], got[0], before[2]], mu, lam)
        assert st == oracle.OK
        for m, want in ((0, Fo[0]), (1, Fs[0])):
            assert np.linalg.norm(got[m] - want) <= 1e-2 * np.linalg.norm(want), m
        return
    # FP32 Grams amplified by the solves, as in the stepwise test
    for m in range(3):
        assert np.linalg.norm(got[m] - Fo[m]) <= 1e-4 * np.linalg.norm(Fo[m]), m
    want = oracle.joint_loss(oy, ot, Fo, mu, lam)
    assert abs(obj - want) <= 1e-5 * abs(want)
