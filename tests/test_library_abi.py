"""The C-ABI library builds, loads and exports every symbol the public header declares (no GPU needed)."""
import ctypes
import os
import re
import subprocess
import sys

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
