"""The order of the MTTKRP's sums: what it may depend on.

BF16 storage turns a last bit of a sum into 2^-9 of a factor entry now and then,
so a BF16 class of a batch takes a walk shape that follows from its rank alone,
never from a timing.
"""
import pytest
import torch

from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu


def bf16_batch(R, dims, nnz, n, autotune=True):
    jobs = []
    for k in range(n):
        idx, val = synth.uniform_tensor(dims, nnz, seed=900 + k, device="cuda")
        t = dfacto.Tensor(idx, val, dims, rank=R, factor_dtype=dfacto.BF16)
        t.set_factors(synth.normal_factors(dims, R, seed=950 + k, device="cuda"))
        jobs.append(t)
    return jobs, dfacto.Batch(jobs, autotune=autotune)


def sweeps(jobs, b, n=2):
    fits = [b.als_iter()[1] for _ in range(n)]
    return [t.factors(torch.bfloat16) for t in jobs], fits


@pytest.mark.parametrize("R", [8, 12, 16, 20, 24, 32])
def test_bf16_batch_shape_follows_from_the_rank(R):
    for dims, nnz, n in (([40, 30, 20], 500, 1), ([300, 200, 100], 20000, 4),
                         ([20000, 10000, 5000], 1200000, 6)):
        jobs, b = bf16_batch(R, dims, nnz, n)
        (c,) = b.classes()
        assert (c.vec, c.seg_nnz) == (8 if R in (24, 32) else 4, 64), (dims, c.vec, c.seg_nnz)
        b.close()


def test_bf16_batches_of_the_same_jobs_agree_bit_for_bit():
    for R in (8, 16, 32):
        got = []
        for _ in range(2):
            jobs, b = bf16_batch(R, [20000, 10000, 5000], 400000, 3)
            got.append(sweeps(jobs, b))
            b.close()
        assert got[0][1] == got[1][1]
        for f0, f1 in zip(got[0][0], got[1][0]):
            assert all(torch.equal(x, y) for x, y in zip(f0, f1)), R


def test_default_segments_hold_no_longer_chain_than_128():
    # enough nonzeros that a rule by size alone would take longer segments
    dims, R = [60000, 50000, 40000], 32
    idx, val = synth.uniform_tensor(dims, 12000000, seed=77, device="cuda")
    F = synth.normal_factors(dims, R, seed=78, device="cuda")
    got = []
    for seg in (0, 128):
        t = dfacto.Tensor(idx, val, dims, rank=R, seg_nnz=seg)
        assert max(dfacto.dfacto_get_info(t.h).seg_nnz) <= 128
        t.set_factors(F)
        got.append([t.mttkrp(m) for m in range(3)])
    assert all(torch.equal(a, b) for a, b in zip(*got))


def test_segments_are_not_cut_short_where_the_sms_have_work():
    # (dims, nonzeros, rank, walk) -> segment length: fibers of 66 to 200 nonzeros,
    # and one lane per segment, where short segments made walk 1 half as fast
    for dims, nnz, R, seg in (([300, 200, 100], 2000000, 16, 128), ([300, 200, 100], 4000000, 32, 128),
                              ([300000, 200000, 100000], 8000000, 1, 128),
                              ([300000, 200000, 100000], 8000000, 4, 128)):
        idx, val = synth.uniform_tensor(dims, nnz, seed=5, device="cuda")
        for walk in (1, 2):
            t = dfacto.Tensor(idx, val, dims, rank=R, walk=walk)
            assert list(dfacto.dfacto_get_info(t.h).seg_nnz) == [seg] * 3
