"""Streaming passes launched back to back, each reading what the one before wrote, on grids on both sides of the size from which a
pass lets its successor's blocks in early: the same bits as with a synchronisation after every call."""
import pytest

pytestmark = pytest.mark.gpu


# tiles of 128 x 128: 1, 144 (under one block per SM), 480 and 512 (either side of the rule), 1024
@pytest.mark.parametrize("d_out,d_in", [(128, 128), (3072, 768), (3840, 2048), (4096, 2048), (4096, 4096)])
def test_chained_passes_wait_for_each_other(d_out, d_in):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()

    def chain(settle):
        W = torch.randn((d_out, d_in), generator=torch.Generator("cuda").manual_seed(5), dtype=torch.bfloat16, device="cuda")
        v, m, k = B.alloc_compressed(d_out, d_in)
        vt, mt, _ = B.alloc_compressed(d_in, d_out)
        k2, D = torch.empty_like(k), torch.empty_like(W)
        for _ in range(3):
            for call in (lambda: B.slope_prune_24(W, v, m, k), lambda: B.slope_double_prune(W, k, vt, mt, k2),
                         lambda: B.slope_apply_mask(W, k, D), lambda: B.slope_sparse_add(v, v, 0.5, 0.25, v),
                         lambda: B.slope_update_sparse_matrix(v, k, mt, vt), lambda: B.slope_double_prune_nm(D, k, 2, 4, W, k2),
                         lambda: B.slope_prune_24_double(W, v, m, k, vt, mt, k2), lambda: B.slope_prune_nm(W, 3, 8, W, k)):
                call()
                if settle:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return W, v, m, k, vt, mt, k2, D

    for a, b in zip(chain(False), chain(True)):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    assert B.slope_poll_status() == 0


@pytest.mark.parametrize("d_out,d_in", [(4096, 4096), (3840, 2560)])
@pytest.mark.parametrize("r", [32, 256])                        # adapter gradients inside the weight-gradient launch / beside it
def test_gradients_wait_for_the_mask(d_out, d_in, r):
    """The weight gradient reads the mask that the pruning pass in front of it writes, in an array that held another mask."""
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    b = 96
    gen = torch.Generator("cuda").manual_seed(7)
    new = lambda *shape: torch.randn(shape, generator=gen, dtype=torch.bfloat16, device="cuda")
    Ws, X, dY, T, dT = [new(d_out, d_in), new(d_out, d_in)], new(b, d_in), new(b, d_out), new(b, r), new(b, r)
    ws = torch.empty(B.slope_bwd_dw_adapter_workspace_bytes(b, d_out, d_in, r), dtype=torch.uint8, device="cuda")

    def chain(settle):
        v, m, k = B.alloc_compressed(d_out, d_in)
        out = []
        for W in Ws * 2:
            dWc, dL, dR = (torch.empty(s, dtype=torch.bfloat16, device="cuda") for s in ((d_out, d_in // 2), (d_in, r), (r, d_out)))
            B.slope_prune_24(W, v, m, k)
            if settle:
                torch.cuda.synchronize()
            B.slope_linear_bwd_dw_adapter(dY, X, T, dT, k, dWc, dL, dR, ws)
            out += [dWc, dL, dR]
        torch.cuda.synchronize()
        return out

    for x, y in zip(chain(False), chain(True)):
        assert torch.equal(x.view(torch.int16), y.view(torch.int16))
    assert B.slope_poll_status() == 0
