"""N:M passes bit for bit against the oracle at the smallest matrix, at odd multiples of 128 in either dimension, and
in place, for every group size, on tie-heavy data (the selection works on pairs of groups packed into
half-words: a carry between them or a wrong tie would show here)."""
import numpy as np
import pytest

from paper_2608_24070_b200 import inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(1, 2), (1, 4), (3, 4), (1, 8), (4, 8), (7, 8), (1, 16), (8, 16), (15, 16)])
@pytest.mark.parametrize("d_out,d_in", [(128, 128), (128, 1152), (1152, 128), (640, 384)])
def test_nm_passes_at_odd_sizes(oracle, n, m, d_out, d_in):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    rng = np.random.Generator(np.random.PCG64(61 + m))
    few = si.f32_to_bf16_bits(np.array([0.0, -0.0, 0.5, -0.5, 1.0, -1.0], np.float32))
    special = np.array([0x7F80, 0xFF80, 0x7FC0, 0x0001, 0x8001, 0x7F7F, 0x8080, 0xFFFF], np.uint16)
    W = np.where(rng.random((d_out, d_in)) < 0.5, rng.choice(few, (d_out, d_in)), rng.choice(special, (d_out, d_in))).astype(np.uint16)
    WR_o, mask1_o = oracle.prune_nm(W, n, m)
    WRC_o, mask2_o = oracle.double_prune_nm(W, mask1_o, n, m)
    A = B.bf16_from_bits(W)
    mask1 = torch.empty((d_out, d_in // 8), dtype=torch.uint8, device="cuda")
    mask2 = torch.empty_like(mask1)
    out = torch.empty_like(A)
    B.slope_prune_nm(A, n, m, out, None)
    assert np.array_equal(B.bits_from_bf16(out), WR_o)
    B.slope_prune_nm(A, n, m, A, mask1)                      # in place
    assert np.array_equal(B.bits_from_bf16(A), WR_o) and np.array_equal(mask1.cpu().numpy(), mask1_o)
    B.slope_double_prune_nm(A, mask1, n, m, A, mask2)
    assert np.array_equal(B.bits_from_bf16(A), WRC_o) and np.array_equal(mask2.cpu().numpy(), mask2_o)
    assert B.slope_poll_status() == 0
