"""Auxiliary streams kept from destroyed handles: by context (the bookkeeping
header, compiled with the host compiler), with two contexts on one device, and
with handles built and destroyed by several threads."""
import os
import shutil
import subprocess
import sys
import threading

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_kept_sets_by_context(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "kept_sets_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread",
                    "-I", os.path.join(ROOT, "paper_1406_4519_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "kept_sets_check.cpp"), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0 and "ALL OK" in res.stdout, res.stdout + res.stderr


# One nonzero and rank 2: no kernel of the build or the MTTKRP needs a shared memory
# opt-in, which is recorded per device.
_TWO_CONTEXTS = """
import ctypes, torch
from paper_1406_4519_gb300 import dfacto
cu = ctypes.CDLL("libcuda.so.1")
def ok(e): assert e == 0, e
ok(cu.cuInit(0))
ctx = [ctypes.c_void_p(), ctypes.c_void_p()]
for c in ctx:
    ok(cu.cuCtxCreate_v2(ctypes.byref(c), 0, 0))
    ok(cu.cuCtxPopCurrent_v2(ctypes.byref(ctypes.c_void_p())))
idx, val = torch.tensor([[1], [2], [3]], dtype=torch.int32), torch.tensor([2.5])
for k in (0, 0, 1, 1, 0, 1):
    ok(cu.cuCtxPushCurrent_v2(ctx[k]))
    t = dfacto.Tensor(idx, val, [4, 5, 6], rank=2, stream=0)
    assert dfacto.dfacto_get_info(t.h).norm_x2 == 6.25
    del t
    ok(cu.cuCtxPopCurrent_v2(ctypes.byref(ctypes.c_void_p())))
print("two contexts ok")
"""


@pytest.mark.gpu
def test_two_contexts_on_one_device():
    res = subprocess.run([sys.executable, "-c", _TWO_CONTEXTS], cwd=ROOT, capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0 and "two contexts ok" in res.stdout, res.stdout + res.stderr


@pytest.mark.gpu
def test_handles_built_and_destroyed_by_several_threads():
    from paper_1406_4519_gb300 import dfacto, synth

    dims = [50, 40, 30]
    idx, val = synth.uniform_tensor(dims, 3000, seed=1, device="cuda")
    F = synth.normal_factors(dims, 8, seed=2, device="cuda")
    torch.cuda.synchronize()

    def fits():
        t = dfacto.Tensor(idx, val, dims, rank=8, stream=torch.cuda.Stream().cuda_stream)
        t.set_factors(F)
        return [t.als_iter()[1] for _ in range(2)], t

    want, first = fits()
    wrong = []

    def work():
        try:
            for _ in range(20):
                got, t = fits()
                if got != want:
                    wrong.append(got)
        except Exception as e:  # reported by the test's own thread
            wrong.append(e)

    th = [threading.Thread(target=work) for _ in range(6)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    assert not wrong, wrong[:3]
