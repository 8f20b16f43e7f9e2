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


# ------------------------------------------------------------------------- every check by itself, on otherwise good arguments
_VIEWS = {"cross": ("q", "k", "v"), "mask": ("q", "k"), "sparse": ("q", "k", "v"), "protected": ("q", "k", "v"),
          "indicators": ("y_v", "yhat_v", "y_a", "yhat_a")}


def _good(name):
    """Arguments of one call that nothing is wrong with: stand-ins on cuda:1, every buffer handed in."""
    def view(i, n=96):
        return _OnGpu((2, 3, n, 64), ptr=4096 * i, stride=(3 * n * 64 + 8, n * 64, 64, 1))

    def f32(i):
        return _OnGpu((2, 3, 2, 2), torch.float32, ptr=4096 * i)

    def feat(i, n):
        return _OnGpu((2, n, 384), ptr=4096 * i)

    u8, ws = _OnGpu((2, 96), torch.uint8, ptr=4096 * 20), _OnGpu((5000,), torch.uint8, ptr=4096 * 30)
    if name == "cross":
        return dict(q=view(1, 32), k=view(2), v=view(3), o=view(4), lse=f32(5), scores=f32(6), score_beta=0.25, score_gamma=0.5,
                    softmax_scale=0.125, ws=ws)
    if name == "mask":
        return dict(q=view(1), k=view(2), scores=f32(3), n_protect=7, k_keep=2, blk=64, flags=0x8001, softmax_scale=0.25,
                    out=dict(block_scores=f32(4), col_idx=f32(5), col_cnt=f32(6), prot_tok=u8, prot_blk=f32(7)), ws=ws)
    if name == "sparse":
        return dict(q=view(1), k=view(2), v=view(3), col_idx=f32(4), col_cnt=f32(5), blk=64, softmax_scale=0.5, o=view(6), lse=f32(7),
                    ws=ws)
    if name == "protected":
        return dict(q=view(1), k=view(2), v=view(3), prot_tok=u8, n_protect=9, blk=64, o=view(6), lse=f32(7), softmax_scale=0.5, ws=ws)
    return dict(y_v=feat(1, 40), yhat_v=feat(2, 40), y_a=feat(3, 24), yhat_a=feat(4, 24), prot_tok=u8, s_cur=f32(5), s_anchor=f32(6),
                lambda_p=0.5, lambda_s=0.25, tau=0.125, eps=0.0625, out=f32(7), ws=ws)


_ENTRY = {"cross": av.avsa_cross_attn_scores, "mask": av.avsa_build_block_mask, "sparse": av.avsa_sparse_self_attn,
          "protected": av.avsa_protected_rows_attn, "indicators": av.avsa_cache_indicators}


def _at(i, n=96):
    return (4096 * i, 3 * n * 64 + 8, n * 64, 64)


_P = [4096 * i for i in range(8)]
_FLAGS, _WS = 4096 * 20, [4096 * 30, 5000, 4097]      # workspace, its size, the stream of cuda:1


@pytest.mark.parametrize("name,want", [
    ("cross", [2, 3, 32, 96, 64, _at(1, 32), _at(2), _at(3), _P[4], _P[5], _P[6], 0.25, 0.5, 0.125]),
    ("mask", [2, 3, 96, 64, 64, _at(1), _at(2), _P[3], 7, 2, 0x8001, 0.25, _P[4], _P[5], _P[6], _FLAGS, _P[7]]),
    ("sparse", [2, 3, 96, 64, 64, _at(1), _at(2), _at(3), _P[4], _P[5], _P[6], _P[7], 0.5]),
    ("protected", [2, 3, 96, 64, 64, _at(1), _at(2), _at(3), _FLAGS, 9, _P[6], _P[7], 0.5]),
    ("indicators", [2, 40, 24, 384, _P[1], _P[2], _P[3], _P[4], _FLAGS, _P[5], _P[6], 0.5, 0.25, 0.125, 0.0625, _P[7]]),
])
def test_good_arguments_reach_the_library_as_they_are(recorded, name, want):
    """Sizes, pointers, strides, counts, the workspace's size and the stream of the tensors' device, in the library's order."""
    _ENTRY[name](**_good(name))
    assert recorded == [(name, want + _WS)]


def _wrong(t, what):
    if what == "none":
        return None
    new = _OnGpu(t.shape, t.dtype, t.stride(), t.data_ptr())
    if what == "fp32":
        new.dtype = torch.float32
    elif what == "host":
        new.is_cuda = False
    elif what == "rank":
        new.shape, new._stride = new.shape[1:], new._stride[1:]
    else:      # the innermost axis not contiguous
        new._stride = new._stride[:-1] + (2,)
    return new


@pytest.mark.parametrize("what,error,match", [
    ("fp32", ValueError, "bf16"), ("host", ValueError, "CUDA"), ("stride", ValueError, "contiguous"),
    ("rank", ValueError, "bf16 tensor|dimensions|unpack"), ("none", AttributeError, "NoneType")])
@pytest.mark.parametrize("name,arg", [(n, a) for n in _VIEWS for a in _VIEWS[n]])
def test_one_wrong_tensor_is_refused(recorded, name, arg, what, error, match):
    """Exactly one property of one tensor is wrong, so that only the check meant for it can refuse the call."""
    args = _good(name)
    if name == "indicators" and what == "rank" and arg != "y_v":
        pytest.skip("any rank is taken there")
    if name == "mask" and what == "none":
        args[arg] = None      # a null view: the library says whether the flags allow it
        if arg == "q":
            args["shape"] = (2, 3, 96, 64)
            args["block_scores"] = args["out"]["block_scores"]
        _ENTRY[name](**args)
        assert recorded.pop()[1][5 + (arg == "k")] == (None, 0, 0, 0)
        return
    args[arg] = _wrong(args[arg], what)
    with pytest.raises(error, match=match):
        _ENTRY[name](**args)
    assert recorded == []
