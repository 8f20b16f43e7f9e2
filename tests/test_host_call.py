"""The marshalling extension refuses what the library could not describe (no GPU needed: nothing is launched)."""
import pytest
import torch

from paper_2608_15522_b200 import binding as av


def _calls(t):
    ws = torch.empty(256, dtype=torch.uint8)
    return {"cross": lambda: av.avsa_cross_attn_scores(t, t, t, o=t, lse=t, scores=t, ws=ws),
            "mask": lambda: av.avsa_build_block_mask(t, t, None, 0, 1, 64, ws=ws),
            "sparse": lambda: av.avsa_sparse_self_attn(t, t, t, t, t, 64, o=t, ws=ws),
            "protected": lambda: av.avsa_protected_rows_attn(t, t, t, t, 1, 64, t, ws=ws),
            "indicators": lambda: av.avsa_cache_indicators(t[0], t[0], t[0], t[0], out=t, ws=ws)}


@pytest.mark.parametrize("name", ["cross", "mask", "sparse", "protected", "indicators"])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_tensors_off_the_gpu_or_of_another_type_are_refused(name, dtype):
    with pytest.raises(ValueError):
        _calls(torch.zeros((1, 2, 64, 64), dtype=dtype))[name]()


@pytest.mark.parametrize("name", ["cross", "mask", "sparse", "protected"])
def test_other_ranks_are_refused(name):
    with pytest.raises(ValueError):
        _calls(torch.zeros((2, 64, 64), dtype=torch.bfloat16))[name]()


def test_missing_tensors_raise_instead_of_reaching_the_library():
    t = torch.zeros((1, 2, 64, 64), dtype=torch.bfloat16)
    for call in (lambda: av.avsa_cross_attn_scores(t, t, None, o=t, lse=t, scores=t, ws=t),
                 lambda: av.avsa_sparse_self_attn(None, t, t, t, t, 64, o=t, ws=t)):
        with pytest.raises((AttributeError, ValueError)):
            call()
