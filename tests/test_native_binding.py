"""The binding's native marshalling refuses what it cannot hand to the C ABI, before anything is launched."""
import pytest
import torch


@pytest.fixture(scope="module")
def B():
    from paper_2608_24070_b200 import binding, build

    build.build()
    binding.lib()
    return binding


def test_only_contiguous_cuda_tensors_are_taken(B):
    W = torch.zeros(128, 128, dtype=torch.bfloat16)
    for call in (lambda: B.slope_prune_24(W, W, W), lambda: B.slope_linear_fwd(W, W, W, 128, W),
                 lambda: B.slope_adapter_fwd_bwd(0, W, None, W, None, 1, 128, 128, 16, T=W)):
        with pytest.raises(AssertionError, match="contiguous CUDA tensors"):
            call()


def test_arguments_of_the_wrong_kind(B):
    with pytest.raises(TypeError):
        B.slope_prune_24(None, None, None)
    with pytest.raises(TypeError):
        B.slope_dense_linear_fwd(1, 2, 3)
    with pytest.raises((TypeError, OverflowError)):
        B.slope_adapter_fwd_bwd(1 << 40, None, None, None, None, 1, 128, 128, 16)


@pytest.mark.gpu
def test_statuses_of_the_library_become_errors(B):
    with pytest.raises(B.SlopeError) as e:                       # all pointers missing: refused by the argument checks
        B.slope_adapter_fwd_bwd(0, None, None, None, None, 1, 128, 128, 16)
    assert e.value.status == 1


def test_a_module_built_against_another_torch_is_neither_kept_nor_loaded(B, monkeypatch):
    from paper_2608_24070_b200 import build

    assert build.up_to_date()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert not build.up_to_date()
    monkeypatch.setattr(B, "_lib", None)
    with pytest.raises(RuntimeError, match="another torch"):
        B.lib()
