"""Padded factor copies stay in step with the factors through every call that
changes one, and the CSR build at the sizes where its scans and its digit
widths change."""
import numpy as np
import pytest
import torch

import oracle
from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu

DIMS = [300, 200, 150]


def tensor(R, dtype, seed=3100, **kw):
    idx, val = synth.uniform_tensor(DIMS, 20000, seed=seed, device="cuda")
    t = dfacto.Tensor(idx, val, DIMS, rank=R, factor_dtype=dtype, **kw)
    t.set_factors(synth.normal_factors(DIMS, R, seed + 1, "cuda"))
    return t, idx, val


def check_fresh(t, idx, val, R, dtype):
    """The handle's MTTKRPs are those of a new handle with the same factors, bit
    for bit: the same kernels on the same values."""
    u = dfacto.Tensor(idx, val, DIMS, rank=R, factor_dtype=dtype)
    u.set_factors(t.factors())
    for m in range(3):
        assert torch.equal(t.mttkrp(m), u.mttkrp(m)), m


@pytest.mark.parametrize("dtype", [dfacto.F32, dfacto.BF16])
@pytest.mark.parametrize("R", [3, 10, 12, 13, 30])
def test_padded_copies_follow_the_factors(R, dtype):
    t, idx, val = tensor(R, dtype, lambda_reg=0.1)
    check_fresh(t, idx, val, R, dtype)
    for _ in range(2):
        t.als_iter()
        check_fresh(t, idx, val, R, dtype)
    dfacto.dfacto_set_factors(t.h, 1, synth.normal_factors(DIMS, R, 77, "cuda")[1])
    check_fresh(t, idx, val, R, dtype)
    t.gd_iter()
    check_fresh(t, idx, val, R, dtype)
    u, v = torch.meshgrid(torch.arange(0, 300, 7), torch.arange(0, 200, 9), indexing="ij")
    yidx = torch.stack([u.reshape(-1), v.reshape(-1)]).to(torch.int32).cuda().contiguous()
    t.set_ratings(yidx, torch.ones(yidx.shape[1], device="cuda"), 0.5)
    t.joint_als_iter()
    check_fresh(t, idx, val, R, dtype)
    t.joint_gd_iter()
    check_fresh(t, idx, val, R, dtype)


@pytest.mark.parametrize("dtype", [dfacto.F32, dfacto.BF16])
def test_padded_copies_follow_a_batch(dtype):
    R = 10
    jobs = [tensor(R, dtype, seed=s) for s in (3200, 3300)]
    for t, idx, val in jobs:
        check_fresh(t, idx, val, R, dtype)  # the copies exist before the batch
    b = dfacto.Batch([j[0] for j in jobs], autotune=False)
    for _ in range(3):  # issued, captured, replayed
        b.als_iter()
        for t, idx, val in jobs:
            check_fresh(t, idx, val, R, dtype)
    b.close()
    for t, idx, val in jobs:
        check_fresh(t, idx, val, R, dtype)


# Tile counts of a digit and words of 32 nonzeros are scanned by one block up to
# 65,536 values (2,097,152 nonzeros); nine-bit digits
# are weighed differently above 4,194,304 nonzeros.
@pytest.mark.parametrize("nnz", [65535, 65536, 65537, 2097152, 2097153, 2097185, 4194304, 4194305])
def test_csr_bit_exact_at_scan_and_digit_limits(nnz):
    dims = [3000, 700, 260]
    idx, val = synth.uniform_tensor(dims, nnz, seed=3400, device="cuda")
    t = dfacto.Tensor(idx, val, dims, rank=4)
    ot = oracle.Tensor(idx.cpu().numpy(), val.cpu().numpy(), dims)
    for m in range(3):
        st, want = oracle.build_csr(ot, m)
        assert st == oracle.OK
        got = t.csr(m)
        assert got["nfib"] == want["nfib"]
        for key in ("fiber_ptr", "fiber_idx", "nz_ptr", "nz_idx"):
            np.testing.assert_array_equal(got[key].cpu().numpy(), want[key], err_msg="%s %d" % (key, m))
        np.testing.assert_array_equal(got["nz_val"].cpu().numpy().view(np.uint32),
                                      want["nz_val"].view(np.uint32))
