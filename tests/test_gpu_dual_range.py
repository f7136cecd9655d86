"""The line search's walk over the nonzeros where a value times a gradient's scale
leaves the range of FP32, though the value times the scaled gradient does not:
factors A and C of 1e-20 and values near 1e4 make B's gradient about 1e-36, so its
scale is about 1e36."""
import math

import pytest
import torch

from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("line_search", [0, 1])
@pytest.mark.parametrize("R", [1, 2, 8, 10])
def test_small_gradients_next_to_large_values(R, line_search):
    dims = [40, 30, 20]
    idx, val = synth.uniform_tensor(dims, 2000, seed=6, device="cuda")
    val = 1e4 * (1 + val)
    A, B, C = synth.normal_factors(dims, R, seed=7, device="cuda")
    got = []
    for walk in (1, 2):
        t = dfacto.Tensor(idx, val, dims, rank=R, walk=walk, line_search=line_search)
        t.set_factors([A * 1e-20, B, C * 1e-20])
        st, loss, alpha = t.gd_iter()
        assert st == dfacto.OK and math.isfinite(loss) and alpha > 0, (walk, st, loss, alpha)
        got.append((loss, alpha, t.factors()))
    # walk 1 and walk 2 add the terms in different orders: FP32 sums of 2,000 values
    assert abs(got[0][0] - got[1][0]) <= 1e-5 * abs(got[0][0])
    assert abs(got[0][1] - got[1][1]) <= 1e-5 * got[0][1]
