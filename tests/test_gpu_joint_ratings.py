"""The ratings term of the joint objective adds a rating's products as a tree over
the padded rank: FP32 products, then halves added until one is left.  Formed here
the same way, so what is left between the two is FP64 rounding."""
import numpy as np
import pytest
import torch

from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu


def tree_dot(a, b):
    R = a.shape[-1]
    RP = 8 if R <= 8 else 16 if R <= 16 else 32
    v = np.zeros(a.shape[:-1] + (RP,), np.float32)
    v[..., :R] = a * b
    while v.shape[-1] > 1:
        h = v.shape[-1] // 2
        v = v[..., :h] + v[..., h:]
    return v[..., 0]


@pytest.mark.parametrize("dtype", [dfacto.F32, dfacto.BF16])
@pytest.mark.parametrize("R", [1, 5, 8, 10, 16, 17, 32])
def test_ratings_loss_is_the_tree_sum(R, dtype):
    dims = [300, 40, 20]
    g = torch.Generator().manual_seed(5 + R)
    yidx = torch.stack([torch.arange(300), torch.randint(0, 40, (300,), generator=g)]).to(torch.int32)
    yval = torch.zeros(300)  # every residual is the dot product itself
    idx, val = synth.uniform_tensor(dims, 500, seed=3, device="cuda")
    t = dfacto.Tensor(idx, val, dims, rank=R, factor_dtype=dtype)
    F = [1 + 0.1 * f for f in synth.normal_factors(dims, R, seed=4, device="cuda")]
    t.set_factors([f.bfloat16() if dtype == dfacto.BF16 else f for f in F])
    t.set_ratings(yidx.cuda(), yval.cuda(), 0.0)  # mu = 0, lambda = 0: the ratings term alone
    A, B, _ = [f.cpu().numpy() for f in t.factors()]
    u = tree_dot(A[yidx[0]], B[yidx[1]]).astype(np.float64)
    want = 0.5 * float((u * u).sum())
    # 300 FP64 terms on each side
    assert abs(t.joint_objective() - want) <= 300 * 2.3e-16 * want
