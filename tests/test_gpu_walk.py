"""MTTKRP walk 2 against walk 1 (bit for bit) and the FP64 oracle at the sizes
where its batches, segments and buffers end: nonzero counts around 32 and around
a segment, rows of one nonzero and rows longer than a segment, every lane layout
the default shapes use, both storage types."""
import numpy as np
import pytest
import torch

import oracle
from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu

# FP32 sums over segments of at most 256 nonzeros, normwise (as the parity tests).
TOL = 1e-5

SHAPES = [  # dims, nonzeros
    ([3, 2, 7], 1), ([40, 30, 20], 31), ([40, 30, 20], 32), ([40, 30, 20], 33),
    ([1, 50, 60], 257), ([700, 1, 1], 513), ([5000, 40, 40], 4096), ([60, 50, 40], 20001),
    ([3000, 2000, 1000], 40960),
]


@pytest.mark.parametrize("dtype", [dfacto.F32, dfacto.BF16])
@pytest.mark.parametrize("R", [1, 2, 4, 6, 8, 10, 16, 24, 32, 40, 64, 128])
def test_walks_agree_bitwise(R, dtype):
    for n, (dims, nnz) in enumerate(SHAPES):
        idx, val = synth.uniform_tensor(dims, min(nnz, dims[0] * dims[1] * dims[2]), 900 + n, "cuda")
        F = synth.normal_factors(dims, R, 950 + n, "cuda")
        if dtype == dfacto.BF16:
            F = [f.to(torch.bfloat16) for f in F]
        ot = oracle.Tensor(idx.cpu().numpy(), val.cpu().numpy(), dims)
        Fh = [f.double().cpu().numpy() for f in F]
        for seg in (0, 256):
            got = []
            for walk in (1, 2):
                t = dfacto.Tensor(idx, val, dims, rank=R, factor_dtype=dtype, seg_nnz=seg, walk=walk)
                t.set_factors(F)
                got.append([t.mttkrp(m) for m in range(3)])
            for m in range(3):
                assert torch.equal(got[0][m], got[1][m]), (dims, nnz, R, seg, m)
                want = oracle.mttkrp(ot, m, Fh)
                err = np.linalg.norm(got[1][m].double().cpu().numpy() - want) / np.linalg.norm(want)
                assert err <= TOL, (dims, nnz, R, seg, m, err)
