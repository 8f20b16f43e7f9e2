"""The marshalling extension refuses what the library could not describe (no GPU needed: nothing is launched)."""
import ctypes

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


# ------------------------------------------------------------------------- the library's entry points replaced by recorders
_i, _f, _p, _sz, _u, _T = ctypes.c_int, ctypes.c_float, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_uint, av._Bf16Tensor4
_SIGNATURES = {
    "cross": [_i] * 5 + [_T] * 3 + [_p] * 3 + [_f] * 3 + [_p, _sz, _p],
    "mask": [_i] * 5 + [_T] * 2 + [_p, _i, _i, _u, _f] + [_p] * 6 + [_sz, _p],
    "sparse": [_i] * 5 + [_T] * 3 + [_p] * 4 + [_f, _p, _sz, _p],
    "protected": [_i] * 5 + [_T] * 3 + [_p, _i, _p, _p, _f, _p, _sz, _p],
    "indicators": [_i] * 4 + [_p] * 7 + [_f] * 4 + [_p, _p, _sz, _p],
}


@pytest.fixture
def recorded():
    """The extension bound to recorders instead of the library: calls[...] is what would have been called, with what."""
    calls, keep = [], []

    def recorder(name, types):
        def entry(*args):
            calls.append((name, [(a.ptr, a.stride_b, a.stride_h, a.stride_n) if isinstance(a, _T) else a for a in args]))
            return 0
        keep.append(ctypes.CFUNCTYPE(_i, *types)(entry))
        return ctypes.cast(keep[-1], _p).value

    host = av._host()
    host.bind(*(recorder(n, t) for n, t in _SIGNATURES.items()), torch.bfloat16, lambda device: 4096 + device)
    yield calls
    av._host_module = None      # bound to the library again
    av._host()


def test_given_block_scores_in_host_memory_are_refused(recorded):
    """Without q and k the block scores say which device the call runs on; in host memory there is none, and the kernels
    would be handed host pointers."""
    bs = torch.zeros((1, 2, 4, 4))
    with pytest.raises(ValueError, match="CUDA device"):
        av.avsa_build_block_mask(None, None, None, 0, 1, 64, flags=av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES,
                                 block_scores=bs, shape=(1, 2, 256, 64))
    assert recorded == []


class _OnGpu:
    """Stands for a tensor on cuda:1: what the marshalling reads of one, without the device."""

    device = torch.device("cuda", 1)

    def __init__(self, shape, dtype=torch.bfloat16, stride=None, ptr=65536, is_cuda=True):
        self.shape, self.dtype, self.is_cuda, self._ptr = torch.Size(shape), dtype, is_cuda, ptr
        dense, n = [], 1
        for s in reversed(self.shape):
            dense.insert(0, n)
            n *= s
        self._dense, self._n, self._stride = tuple(dense), n, tuple(dense) if stride is None else tuple(stride)

    def stride(self):
        return self._stride

    def data_ptr(self):
        return self._ptr

    def numel(self):
        return self._n

    def get_device(self):
        return 1 if self.is_cuda else -1

    def is_contiguous(self):
        return self._stride == self._dense


def test_a_block_size_that_is_no_integer_is_refused(recorded):
    t, f32, u8, ws = _OnGpu((1, 2, 256, 64)), _OnGpu((1, 2, 4, 4), torch.float32), _OnGpu((1, 256), torch.uint8), _OnGpu((999,))
    out = dict(block_scores=f32, col_idx=f32, col_cnt=f32, prot_tok=u8, prot_blk=u8)
    for blk in (64.0, 64.9, "64"):
        for call in (lambda: av.avsa_sparse_self_attn(t, t, t, f32, f32, blk, o=t, ws=ws),
                     lambda: av.avsa_protected_rows_attn(t, t, t, u8, 1, blk, t, ws=ws),
                     lambda: av.avsa_build_block_mask(t, t, None, 0, 1, blk, out=out, ws=ws)):
            with pytest.raises(TypeError):
                call()
    assert recorded == []


def test_audio_features_of_any_rank_keep_their_token_axis(recorded):
    """The audio tokens are axis 1 of y_a, whatever the channels behind it are split into (the video stream gives B and C)."""
    y_v, out, ws = _OnGpu((2, 40, 384)), _OnGpu((2, 8), torch.float32), _OnGpu((9999,), torch.uint8)
    for shape in ((2, 24, 384), (2, 24, 3, 128), (2, 24 * 384)):
        y_a = _OnGpu(shape)
        av.avsa_cache_indicators(y_v, y_v, y_a, y_a, out=out, ws=ws)
        assert recorded.pop()[1][:4] == [2, 40, shape[1], 384]
    for bad_v in ((80, 384), (2, 40, 3, 128)):
        with pytest.raises(ValueError):
            av.avsa_cache_indicators(_OnGpu(bad_v), y_v, y_v, y_v, out=out, ws=ws)
    assert recorded == []
