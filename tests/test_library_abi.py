"""The C-ABI library builds, loads and exports every symbol the public header declares (no GPU needed)."""
import ctypes
import os
import re
import subprocess
import sys

import pytest
import torch

from paper_2608_15522_b200 import binding as av
from paper_2608_15522_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "avsa.h")).read()
    return sorted(set(re.findall(r"AVSA_API\s+[\w\s\*]+?\b(avsa_\w+)\s*\(", text)))


def test_header_declares_the_three_calls():
    names = _declared_symbols()
    for n in ("avsa_cross_attn_scores", "avsa_build_block_mask", "avsa_sparse_self_attn"):
        assert n in names and n + "_workspace_bytes" in names


def test_library_builds_loads_and_exports_every_declared_symbol():
    path = build.build_library()
    assert os.path.exists(path)
    lib = ctypes.CDLL(path)
    for name in _declared_symbols():
        assert hasattr(lib, name), name
    assert sorted(av.EXPORTS) == sorted(n for n in _declared_symbols())


def test_host_only_entry_points():
    assert av.avsa_version() >= 100
    assert av.status_string(av.AVSA_OK) == "ok"
    assert "column list" in av.status_string(av.AVSA_ERR_BAD_MASK)
    assert av.avsa_count_from_percent(10, 140) == 14
    assert av.avsa_count_from_percent(5, 32760) == 1638
    assert av.avsa_count_from_percent(25, 256) == 64
    assert av.avsa_count_from_percent(20, 384) == 77
    assert av.avsa_count_from_percent(0, 100) == 0
    assert av.avsa_cross_attn_scores_workspace_bytes(1, 24, 256, 32760, 128) > 0
    assert av.avsa_build_block_mask_workspace_bytes(1, 24, 32760, 128, 128) > 2 * 24 * 256 * 128 * 4
    assert av.avsa_sparse_self_attn_workspace_bytes(1, 24, 32760, 128, 128) >= 16
    assert av.avsa_cross_attn_scores_workspace_bytes(1, 1, 1, 1, 96) == 0


def test_more_pairs_than_32_bits_count_are_refused():
    """2^32 (batch, head) pairs wrap to 0, which the plans of the work divide by: the queries say 0 (not supported) and the calls
    AVSA_ERR_UNSUPPORTED, before any pointer is followed.  In a process of its own: a division by 0 ends it."""
    code = """if True:
        from paper_2608_15522_b200 import binding as av
        for b, h in ((65536, 65536), (40000, 60000)):
            assert av.avsa_cross_attn_scores_workspace_bytes(b, h, 4, 4, 64) == 0
            assert av.avsa_protected_rows_attn_workspace_bytes(b, h, 4, 64, 64, 1) == 0
        lib, t = av.load_library(), av._Bf16Tensor4(4096, 8, 8, 64)
        args = (65535, 65535, 4)
        assert lib.avsa_cross_attn_scores(*args, 4, 64, t, t, t, 4096, 4096, 4096, 0.0, 1.0, 0.0, 4096, 1 << 40, 0) == av.AVSA_ERR_UNSUPPORTED
        assert lib.avsa_protected_rows_attn(*args, 64, 64, t, t, t, 4096, 1, 4096, 4096, 0.0, 4096, 1 << 40, 0) == av.AVSA_ERR_UNSUPPORTED
    """
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    assert r.returncode == 0, r.stdout


_T = av._Bf16Tensor4(4096, 64 * 4096, 4096, 64)
_T128 = av._Bf16Tensor4(4096, 128 * 4096, 4096, 128)


def _call(name, ws):
    """A call that nothing is wrong with but, perhaps, the alignment of its workspace."""
    lib, p, big = av.load_library(), 8192, 1 << 40
    cross = lambda nq, nk, t, d, scores: lib.avsa_cross_attn_scores(1, 2, nq, nk, d, t, t, t, p, p, p if scores else None, 0.0, 1.0, 0.0, ws, big, 0)
    mask = lambda n, flags: lib.avsa_build_block_mask(1, 2, n, 64, 64, _T, _T, p, 3, 1, flags, 0.0, p, p, p, p, p, ws, big, 0)
    sparse = lambda n, t, d: lib.avsa_sparse_self_attn(1, 24, n, d, d, t, t, t, p, p, p, p, 0.0, ws, big, 0)
    protected = lambda n_protect: lib.avsa_protected_rows_attn(1, 2, 4096, 128, 128, _T128, _T128, _T128, p, n_protect, p, p, 0.0, ws, big, 0)
    return {"sparse": lambda: sparse(4096, _T128, 128), "sparse_pairs": lambda: sparse(64 * 64, _T, 64),
            "mask": lambda: mask(4096, av.AVSA_PROTECT_ROWS), "mask_select_in_pooling": lambda: mask(500, av.AVSA_PROTECT_ROWS),
            "mask_short": lambda: mask(200, av.AVSA_PROTECT_ROWS), "mask_given": lambda: mask(4096, av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES),
            "cross_few_keys": lambda: cross(4096, 200, _T, 64, True), "cross_parts": lambda: cross(100, 32768, _T, 64, True),
            "cross_whole_rows": lambda: cross(64 * 1024, 300, _T, 64, False), "cross_whole_rows_reverse": lambda: cross(64 * 1024, 300, _T, 64, True),
            "protected_none": lambda: protected(0), "protected_parts": lambda: protected(200),
            "indicators": lambda: lib.avsa_cache_indicators(1, 64, 64, 64, 4096, 4096, 4096, 4096, None, None, None, 0.5, 0.1, 0.2, 1e-6, p, ws, big, 0)}[name]()


@pytest.mark.skipif(torch.cuda.is_available(), reason="the accepted calls would be launched")
@pytest.mark.parametrize("name,needs", [
    ("sparse", 4), ("sparse_pairs", 4), ("mask", 16), ("mask_select_in_pooling", 16), ("mask_short", 4), ("mask_given", 4),
    ("cross_few_keys", 4), ("cross_parts", 32), ("cross_whole_rows", 4), ("cross_whole_rows_reverse", 16), ("protected_none", 4),
    ("protected_parts", 32), ("indicators", 16)])
def test_a_workspace_less_aligned_than_its_accesses_is_refused(name, needs):
    """By every call, before anything is enqueued; where only words of 4 bytes are touched, 4 bytes are enough."""
    for offset in (1, 2, 4, 8, 16, 32):
        refused = _call(name, (1 << 20) + offset) == av.AVSA_ERR_INVALID_ARG
        assert refused == (offset % needs != 0), offset
