"""Calls recorded into a CUDA graph by the caller: a replay works on the factors of
its own time, also at ranks whose factors the walk reads through padded copies."""
import pytest
import torch

from paper_1406_4519_gb300 import dfacto, synth

pytestmark = pytest.mark.gpu

DIMS = [400, 300, 200]


def handle(R, dtype, stream, seed=7):
    idx, val = synth.uniform_tensor(DIMS, 20000, seed=6, device="cuda")
    F = [f.abs() for f in synth.normal_factors(DIMS, R, seed=seed, device="cuda")]
    torch.cuda.synchronize()
    t = dfacto.Tensor(idx, val, DIMS, rank=R, factor_dtype=dtype, stream=stream)
    t.set_factors(F)
    return t


def mttkrps(t, out):
    for m in range(3):
        t.mttkrp(m, out[m])


@pytest.mark.parametrize("dtype", [dfacto.F32, dfacto.BF16])
@pytest.mark.parametrize("R", [3, 10, 16, 30])
def test_replayed_mttkrp_reads_the_present_factors(R, dtype):
    s = torch.cuda.Stream()
    t = handle(R, dtype, s)
    out = [torch.empty(d, R, device="cuda") for d in DIMS]
    torch.cuda.synchronize()
    mttkrps(t, out)  # allocates what the calls keep
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        mttkrps(t, out)
    for seed in (8, 9):
        F = synth.normal_factors(DIMS, R, seed=seed, device="cuda")
        torch.cuda.synchronize()
        t.set_factors(F)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        want = [torch.empty_like(o) for o in out]
        twin = handle(R, dtype, s)
        twin.set_factors(F)
        mttkrps(twin, want)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, want)), seed
        direct = [torch.empty_like(o) for o in out]
        mttkrps(t, direct)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(direct, want)), seed


@pytest.mark.parametrize("step", ["gd", "als"])
@pytest.mark.parametrize("R", [10, 16])
def test_replayed_steps_and_direct_calls_between_them(R, step):
    s = torch.cuda.Stream()
    t, twin = handle(R, dfacto.F32, s), handle(R, dfacto.F32, s)
    out = [torch.empty(d, R, device="cuda") for d in DIMS]
    want = [torch.empty(d, R, device="cuda") for d in DIMS]
    torch.cuda.synchronize()

    def one(h):
        (h.gd_iter if step == "gd" else h.als_iter)(False)

    for h, o in ((t, out), (twin, want)):
        one(h)
        mttkrps(h, o)  # padded copies of every factor are up to date here
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        one(t)
    for k in range(4):
        g.replay()
        one(twin)
        if k != 1:
            torch.cuda.synchronize()
            mttkrps(t, out)
            mttkrps(twin, want)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(t.factors(), twin.factors())), k
        assert all(torch.equal(a, b) for a, b in zip(out, want)), k
