"""An infinite or NaN nonzero at a rank the walk pads: the row passes read the
padded MTTKRP rows, whose extra columns are then NaN, and must give what they give
from unpadded rows (an explicit lane width)."""
import numpy as np
import pytest
import torch

from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu


def kinds(x):
    x = x.double().cpu()
    return torch.isnan(x).int() + 2 * torch.isposinf(x).int() + 4 * torch.isneginf(x).int() + 8 * (x == 0).int()


@pytest.mark.parametrize("dtype", [dfacto.F32, dfacto.BF16])
@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("R", [3, 5, 6, 7, 10, 13, 15, 30, 31])
def test_padded_rank_with_a_nonfinite_value(R, bad, dtype):
    dims = [400, 300, 200]
    idx, val = synth.uniform_tensor(dims, 3000, seed=6, device="cuda")
    val = val.clone()
    val[7] = bad
    F = synth.normal_factors(dims, R, seed=7, device="cuda")
    for step in ("als", "gd"):
        got = []
        for vec in (0, 1):
            t = dfacto.Tensor(idx, val, dims, rank=R, factor_dtype=dtype, vec=vec)
            t.set_factors(F)
            if step == "als":
                t.als_iter()
            else:
                t.gd_iter()
            got.append([kinds(f) for f in t.factors()] + [kinds(torch.as_tensor(np.asarray(t.lam())))])
        for m, (a, b) in enumerate(zip(*got)):
            assert torch.equal(a, b), (step, m, int((a != b).sum()))
