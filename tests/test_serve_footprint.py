"""The admission estimate against the arrays a served job holds."""
import pytest
import torch

from paper_1406_4519_gb300 import dfacto, serve, synth


def test_estimate_covers_one_nonzero_per_fiber_in_a_batch():
    n, dims, R = 50_000_000, [20000, 20000, 20000], 8
    words = -(-n // 32)
    copy = 0
    for d in dims:
        copy += 4 * n + 4 * n + 8 * (n + 1) + 4 * (n + 1) + 4 * n  # nz_idx, nz_val, nz_ptr, fiber_idx, fiber_row
        copy += 2 * 4 * words + 4 * -(-n // 128) + 8 * (d + 1)      # end and row bits, segment starts, fiber_ptr
    held = 2 * copy + 2 * R * sum(dims)
    assert serve.footprint_bytes(dims, n, R, 2) >= held


def test_estimate_covers_padded_copies_of_a_long_mode():
    n, dims, R = 1000, [4_000_000, 10, 10], 5
    sd, top = sum(dims), max(dims)
    held = 8 * sd + 2 * R * sd + 4 * R * top + 4 * 8 * (sd + top)  # row pointers, factors, N, padded copies
    assert serve.footprint_bytes(dims, n, R, 2) >= held


@pytest.mark.gpu
@pytest.mark.parametrize("dims,nnz,R", [([4_000_000, 10, 10], 1000, 5), ([4000, 3000, 2000], 2_000_000, 10),
                                        ([30000, 20000, 10000], 1_000_000, 16)])
def test_estimate_covers_what_a_handle_reports(dims, nnz, R):
    idx, val = synth.uniform_tensor(dims, nnz, seed=1, device="cuda")
    t = dfacto.Tensor(idx, val, dims, rank=R, factor_dtype=dfacto.BF16)
    t.set_factors(synth.normal_factors(dims, R, seed=2, device="cuda"))
    t.als_iter()
    assert dfacto.dfacto_get_info(t.h).device_bytes <= serve.footprint_bytes(dims, nnz, R, 2)
