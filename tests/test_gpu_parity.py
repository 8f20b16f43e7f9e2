"""GPU parity: every call of the C ABI against the fp64 CPU oracle on the same seeded inputs.

Bars: integer outputs (flags, lists, counts) bit-exact given the same fp32 score tensors.
bf16 attention outputs O: relative-L2 5e-3 and max-abs 1e-2, the latter scaled by |value| above 1 (the bf16
grid itself is coarser than 1e-2 there).  fp32 log-sum-exps: max-abs 1e-3, unscaled.  fp32 response scores
(Eq. 2): every element within 1e-3 of its own value (plus 1e-6 of the largest score), so that a few wrong
columns cannot hide in a norm.
"""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import avsa_oracle as orc
from paper_2608_15522_b200 import binding as av
from paper_2608_15522_b200 import workloads as wl
from parity_bars import close_lse as _close_lse, close_o as _close, close_scores as _close_scores, np64 as _np64

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _status_ok(ws):
    code, detail = av.avsa_read_status(ws)
    assert code == av.AVSA_OK, f"device status {code} {av.status_string(code)} detail {detail}"


def _oracle_mask(w, q, k, scores64, n_protect, k_keep, flags=av.AVSA_PROTECT_ROWS):
    """Oracle block scores (rounded to fp32, the tensor both sides select from) and its lists."""
    bs32 = orc.block_scores(_np64(q), _np64(k), w.blk).astype(np.float32)
    s32 = scores64.astype(np.float32)
    idx, cnt, ptok, pblk = orc.build_block_mask(bs32, s32, n_protect, k_keep, w.blk, w.n_video,
                                                bool(flags & av.AVSA_PROTECT_ROWS), bool(flags & av.AVSA_PROTECT_COLS))
    return bs32, s32, idx, cnt, ptok, pblk


def _oracle_scores(w, seed):
    qa, kc, vc = wl.make_cross_qkv(w, seed)
    o, lse, A = orc.cross_attention(_np64(qa), _np64(kc), _np64(vc))
    s = orc.column_scores(A, gamma=1.0 / (w.H * w.n_audio))
    return (qa, kc, vc), o, lse, s


# ------------------------------------------------------------------------------------------- mask
@pytest.mark.parametrize("name,flags", [("tiny", 1), ("small128", 1), ("medium128", 1), ("medium128", 3)])
def test_mask_lists_bit_exact_given_oracle_scores(name, flags):
    w = wl.WORKLOADS[name]
    q, k, _ = wl.make_self_qkv(w, 0)
    _, _, _, s64 = _oracle_scores(w, 0)
    n_protect = orc.ceil_pct(w.protect_pct, w.n_video)
    k_keep = max(1, orc.ceil_pct(w.keep_pct, w.n_blocks))
    assert n_protect == av.avsa_count_from_percent(w.protect_pct, w.n_video)
    assert k_keep == max(1, av.avsa_count_from_percent(w.keep_pct, w.n_blocks))
    bs32, s32, idx, cnt, ptok, pblk = _oracle_mask(w, q, k, s64, n_protect, k_keep, flags)
    out = av.avsa_build_block_mask(None, None, torch.from_numpy(s32).cuda(), n_protect, k_keep, w.blk,
                                   flags=flags | av.AVSA_USE_GIVEN_BLOCK_SCORES,
                                   block_scores=torch.from_numpy(bs32).cuda(), shape=(w.B, w.H, w.n_video, w.d))
    _status_ok(out["ws"])
    assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok)
    assert np.array_equal(out["prot_blk"].cpu().numpy(), pblk)
    assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(out["col_idx"].cpu().numpy(), idx)


@pytest.mark.parametrize("name,min_tokens", [("tiny", 3), ("medium128", 2), ("medium128", 16), ("medium128", 128)])
def test_mask_min_tokens_per_block_bit_exact(name, min_tokens):
    """A block counts as protected only from `min_tokens` protected tokens on (flag bits 8-15)."""
    w = wl.WORKLOADS[name]
    _, _, _, s64 = _oracle_scores(w, 0)
    q, k, _ = wl.make_self_qkv(w, 0)
    n_protect = orc.ceil_pct(w.protect_pct, w.n_video)
    k_keep = max(1, orc.ceil_pct(w.keep_pct, w.n_blocks))
    bs32 = orc.block_scores(_np64(q), _np64(k), w.blk).astype(np.float32)
    s32 = s64.astype(np.float32)
    idx, cnt, ptok, pblk = orc.build_block_mask(bs32, s32, n_protect, k_keep, w.blk, w.n_video, True, False,
                                                min_tokens=min_tokens)
    any_blk = orc.protected_blocks(ptok, w.blk)
    if name == "medium128" and min_tokens >= 16:
        assert pblk.sum() < any_blk.sum()      # the threshold bites on these inputs
    out = av.avsa_build_block_mask(None, None, torch.from_numpy(s32).cuda(), n_protect, k_keep, w.blk,
                                   flags=av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES |
                                   av.AVSA_MIN_TOKENS_PER_BLOCK(min_tokens),
                                   block_scores=torch.from_numpy(bs32).cuda(), shape=(w.B, w.H, w.n_video, w.d))
    _status_ok(out["ws"])
    assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok)
    assert np.array_equal(out["prot_blk"].cpu().numpy(), pblk)
    assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(out["col_idx"].cpu().numpy(), idx)


@pytest.mark.parametrize("name,n_blocks,extra", [("tiny", 1, 0), ("medium128", 3, 0), ("medium128", 5, 2),
                                                 ("medium128", 0, 0), ("medium128", 17, 0)])
def test_mask_block_sum_protection_bit_exact(name, n_blocks, extra):
    """Protected blocks = the n blocks with the largest summed response (flag AVSA_PROTECT_BLOCK_SUM), also with
    key-column protection on top (extra = AVSA_PROTECT_COLS).  Block flags, token flags and lists bit-exact."""
    w = wl.WORKLOADS[name]
    _, _, _, s64 = _oracle_scores(w, 0)
    q, k, _ = wl.make_self_qkv(w, 0)
    k_keep = max(1, orc.ceil_pct(w.keep_pct, w.n_blocks))
    bs32 = orc.block_scores(_np64(q), _np64(k), w.blk).astype(np.float32)
    s32 = s64.astype(np.float32)
    s32[:, 5] = np.nan                                   # a NaN score poisons its block's sum: that block ranks last
    idx, cnt, ptok, pblk = orc.build_block_mask(bs32, s32, n_blocks, k_keep, w.blk, w.n_video, True, bool(extra),
                                                block_sum=True)
    assert pblk.sum() == n_blocks * w.B and (n_blocks == w.n_blocks or pblk[:, 0].sum() == 0)
    out = av.avsa_build_block_mask(None, None, torch.from_numpy(s32).cuda(), n_blocks, k_keep, w.blk,
                                   flags=av.AVSA_PROTECT_ROWS | extra | av.AVSA_USE_GIVEN_BLOCK_SCORES |
                                   av.AVSA_PROTECT_BLOCK_SUM,
                                   block_scores=torch.from_numpy(bs32).cuda(), shape=(w.B, w.H, w.n_video, w.d))
    _status_ok(out["ws"])
    assert np.array_equal(out["prot_blk"].cpu().numpy(), pblk)
    assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok)
    assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(out["col_idx"].cpu().numpy(), idx)


def test_mask_ties_nan_and_signed_zero_bit_exact():
    B, H, N, d, blk = 2, 2, 64 * 37 + 5, 64, 64
    NB = (N + blk - 1) // blk
    rng = np.random.default_rng(3)
    bs = rng.integers(-2, 3, size=(B, H, NB, NB)).astype(np.float32)          # heavy ties
    bs[0, 0, 1, :] = 0.0
    bs[0, 0, 2, ::2] = -0.0
    bs[0, 1, 3, 5] = np.nan
    bs[1, 0, 4, :] = np.nan
    bs[1, 1, 5, 7] = np.inf
    bs[1, 1, 5, 9] = -np.inf
    s = rng.integers(0, 4, size=(B, N)).astype(np.float32)
    s[0, 10] = np.nan
    s[1, ::3] = -0.0
    for n_protect, k_keep in ((0, 1), (7, 5), (200, NB), (N, 3), (1, NB - 1)):
        idx, cnt, ptok, pblk = orc.build_block_mask(bs, s, n_protect, k_keep, blk, N)
        out = av.avsa_build_block_mask(None, None, torch.from_numpy(s).cuda(), n_protect, k_keep, blk,
                                       flags=av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES,
                                       block_scores=torch.from_numpy(bs).cuda(), shape=(B, H, N, d))
        _status_ok(out["ws"])
        assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok), (n_protect, k_keep)
        assert np.array_equal(out["prot_blk"].cpu().numpy(), pblk), (n_protect, k_keep)
        assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt), (n_protect, k_keep)
        assert np.array_equal(out["col_idx"].cpu().numpy(), idx), (n_protect, k_keep)


def test_mask_long_sequence_beyond_the_shared_memory_key_cache():
    """N above 57344 tokens: the token select re-reads global memory instead of staging keys on chip."""
    B, H, N, d, blk = 2, 1, 60000 + 77, 128, 128
    NB = (N + blk - 1) // blk
    rng = np.random.default_rng(9)
    bs = rng.standard_normal((B, H, NB, NB)).astype(np.float32)
    s = np.round(rng.standard_normal((B, N)) * 50).astype(np.float32) / 50      # many exact ties
    n_protect, k_keep = 3001, 40
    idx, cnt, ptok, pblk = orc.build_block_mask(bs, s, n_protect, k_keep, blk, N)
    out = av.avsa_build_block_mask(None, None, torch.from_numpy(s).cuda(), n_protect, k_keep, blk,
                                   flags=av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES,
                                   block_scores=torch.from_numpy(bs).cuda(), shape=(B, H, N, d))
    _status_ok(out["ws"])
    assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok)
    assert np.array_equal(out["prot_blk"].cpu().numpy(), pblk)
    assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(out["col_idx"].cpu().numpy(), idx)


@pytest.mark.parametrize("n", [1, 3, 129, 511, 513, 4099, 57344, 57347])
@pytest.mark.parametrize("kind", ["log_normal", "outliers", "constant", "two_values", "one_above", "signs"])
def test_mask_token_select_over_ranges_of_scores(n, kind):
    """The select's bins follow the range that the scores span: narrow and wide ranges, ranges stretched by infinities, one value, ties
    at the edge, both signs; lengths around four tokens a lane, a CTA's step and the keys kept in shared memory; a second batch item
    whose flags may begin at any byte."""
    B, H, d, blk = 2, 1, 128, 128
    NB = (n + blk - 1) // blk
    rng = np.random.default_rng(n)
    s = np.exp(0.3 * rng.standard_normal((B, n))).astype(np.float32)
    if kind == "outliers":
        s[0, 0], s[1, n // 2], s[1, n - 1] = np.inf, -np.inf, 1e-30
    elif kind == "constant":
        s[:] = 0.25
    elif kind == "two_values":
        s = np.where(s > 1.2, np.float32(3.0), np.float32(2.0))
    elif kind == "one_above":
        s = np.full((B, n), 1.0, np.float32)
        s[:, n // 3] = np.nextafter(np.float32(1.0), np.float32(2.0))
    elif kind == "signs":
        s = rng.standard_normal((B, n)).astype(np.float32)
    bs = np.zeros((B, H, NB, NB), np.float32)
    for n_protect in sorted({1, (n + 19) // 20, n // 2 + 1, max(1, n - 1), n}):
        _, _, ptok, pblk = orc.build_block_mask(bs, s, n_protect, 1, blk, n)
        out = av.avsa_build_block_mask(None, None, torch.from_numpy(s).cuda(), n_protect, 1, blk,
                                       flags=av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES,
                                       block_scores=torch.from_numpy(bs).cuda(), shape=(B, H, n, d))
        _status_ok(out["ws"])
        assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok), n_protect
        assert np.array_equal(out["prot_blk"].cpu().numpy(), pblk), n_protect


@pytest.mark.parametrize("name", ["tiny", "small128", "medium128"])
def test_block_scores_and_selection_from_pooled_qk(name):
    w = wl.WORKLOADS[name]
    q, k, _ = wl.make_self_qkv(w, 1)
    _, _, _, s64 = _oracle_scores(w, 1)
    n_protect = orc.ceil_pct(w.protect_pct, w.n_video)
    k_keep = max(1, orc.ceil_pct(w.keep_pct, w.n_blocks))
    s32 = s64.astype(np.float32)
    out = av.avsa_build_block_mask(q.cuda(), k.cuda(), torch.from_numpy(s32).cuda(), n_protect, k_keep, w.blk)
    _status_ok(out["ws"])
    want = orc.block_scores(_np64(q), _np64(k), w.blk)
    got = out["block_scores"].cpu().numpy()
    assert np.abs(got - want).max() <= 1e-4 * max(1.0, np.abs(want).max())
    # the lists are exactly the oracle's when it selects from the very tensor the GPU produced
    idx, cnt, ptok, pblk = orc.build_block_mask(got, s32, n_protect, k_keep, w.blk, w.n_video)
    assert np.array_equal(out["col_idx"].cpu().numpy(), idx)
    assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok)
    # and a valid top-k of the oracle's own fp64 scores up to the fp32 rounding of the scores
    gidx, gcnt = out["col_idx"].cpu().numpy(), out["col_cnt"].cpu().numpy()
    tol = 2e-4 * max(1.0, np.abs(want).max())
    for b in range(w.B):
        for h in range(w.H):
            for i in range(w.n_blocks):
                if pblk[b, i] or k_keep >= w.n_blocks:
                    continue
                kept = gidx[b, h, i, : gcnt[b, h, i]]
                rest = np.setdiff1d(np.arange(w.n_blocks), kept)
                assert want[b, h, i, kept].min() >= want[b, h, i, rest].max() - tol


@pytest.mark.parametrize("nb", [1, 8, 16, 17, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("heads", [2, 80])
def test_block_scores_and_lists_short_rows(nb, heads):
    """Rows around 64, 128 and 256 key blocks (one, two or four tiles a warp, two to eight keys a lane), a strip's rows shared by two
    CTAs (2 heads) and not (80): pooled block scores against the oracle, lists bit-exact given those scores."""
    if heads == 80 and nb > 65:
        pytest.skip("strips outnumber the SMs with two heads of this length already, or the oracle takes long")
    B, d = 1, 64
    N = d * (nb - 1) + 23
    g = torch.Generator().manual_seed(nb)
    q = torch.randn((B, heads, N, d), generator=g).bfloat16()
    k = (torch.randn((B, heads, N, d), generator=g) + 0.5).bfloat16()
    s = torch.rand((B, N), generator=g)
    n_protect, k_keep = max(1, N // 50), max(1, nb // 5)
    out = av.avsa_build_block_mask(q.cuda(), k.cuda(), s.cuda(), n_protect, k_keep, d)
    _status_ok(out["ws"])
    got = out["block_scores"].cpu().numpy()
    want = orc.block_scores(_np64(q), _np64(k), d)
    assert np.abs(got - want).max() <= 1e-4 * max(1.0, np.abs(want).max())
    idx, cnt, ptok, pblk = orc.build_block_mask(got, s.numpy(), n_protect, k_keep, d, N)
    assert np.array_equal(out["col_idx"].cpu().numpy(), idx)
    assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(out["prot_blk"].cpu().numpy(), pblk)


@pytest.mark.parametrize("d,nb,tail", [(128, 520, 5), (64, 300, 17), (128, 33, 0)])
def test_block_scores_and_lists_long_rows(d, nb, tail):
    """Rows of more than 256 and more than 512 key blocks (more keys per lane in the select, larger strips in shared
    memory), a ragged last block, and a block count that is no multiple of the 16-row strip: pooled block scores
    against the oracle, lists bit-exact given those scores."""
    blk = d
    N = blk * (nb - 1) + (tail if tail else blk)
    B, H = 1, 2
    g = torch.Generator().manual_seed(nb)
    q = torch.randn((B, H, N, d), generator=g).bfloat16()
    k = (torch.randn((B, H, N, d), generator=g) + 0.5).bfloat16()
    s = torch.rand((B, N), generator=g)
    n_protect, k_keep = N // 50, max(1, nb // 5)
    out = av.avsa_build_block_mask(q.cuda(), k.cuda(), s.cuda(), n_protect, k_keep, blk)
    _status_ok(out["ws"])
    got = out["block_scores"].cpu().numpy()
    want = orc.block_scores(_np64(q), _np64(k), blk)
    assert got.shape == (B, H, nb, nb)
    assert np.abs(got - want).max() <= 1e-4 * max(1.0, np.abs(want).max())
    idx, cnt, ptok, pblk = orc.build_block_mask(got, s.numpy(), n_protect, k_keep, blk, N)
    assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(out["col_idx"].cpu().numpy(), idx)
    assert np.array_equal(out["prot_tok"].cpu().numpy(), ptok) and np.array_equal(out["prot_blk"].cpu().numpy(), pblk)


# ------------------------------------------------------------------------------------------- sparse attention
def _run_sparse_case(w, seed, idx, cnt, want_lse=True):
    q, k, v = wl.make_self_qkv(w, seed)
    o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(),
                                          torch.from_numpy(cnt).cuda(), w.blk, want_lse=want_lse)
    _status_ok(ws)
    # the workloads' logits stay within a few units of each row's first-tile maximum: every item must come from
    # the fast kernel (the growing-maxima tests cover the recomputation path)
    assert av.avsa_redo_count(ws) == 0
    want_o, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, w.blk)
    _close(_np64(o), want_o, f"{w.name} O")
    if want_lse:
        _close_lse(_np64(lse), want_l, f"{w.name} lse")
    return _np64(o), want_o


@pytest.mark.parametrize("name", ["tiny", "small128", "medium128"])
def test_sparse_attention_matches_oracle_under_protected_mask(name):
    w = wl.WORKLOADS[name]
    q, k, _ = wl.make_self_qkv(w, 0)
    _, _, _, s64 = _oracle_scores(w, 0)
    n_protect = orc.ceil_pct(w.protect_pct, w.n_video)
    k_keep = max(1, orc.ceil_pct(w.keep_pct, w.n_blocks))
    _, _, idx, cnt, _, pblk = _oracle_mask(w, q, k, s64, n_protect, k_keep)
    assert 0 < pblk.sum() < pblk.size or name == "small128"
    _run_sparse_case(w, 0, idx, cnt)


@pytest.mark.parametrize("name", ["tiny", "small128", "medium128"])
def test_sparse_attention_keep_all_is_dense(name):
    w = wl.WORKLOADS[name]
    NB = w.n_blocks
    idx = np.broadcast_to(np.arange(NB, dtype=np.int32), (w.B, w.H, NB, NB)).copy()
    cnt = np.full((w.B, w.H, NB), NB, np.int32)
    got, _ = _run_sparse_case(w, 2, idx, cnt)
    q, k, v = wl.make_self_qkv(w, 2)
    dense, _ = orc.dense_attention(_np64(q), _np64(k), _np64(v))
    _close(got, dense, f"{name} keep-all vs dense")


def test_sparse_attention_single_and_odd_counts():
    """Lists of 1, 2 and 3 entries, and the last (ragged) key block alone."""
    w = wl.WORKLOADS["medium128"]
    NB = w.n_blocks
    idx = np.full((w.B, w.H, NB, NB), -1, np.int32)
    cnt = np.zeros((w.B, w.H, NB), np.int32)
    rng = np.random.default_rng(5)
    for b in range(w.B):
        for h in range(w.H):
            for i in range(NB):
                c = 1 + (i % 3)
                cols = np.sort(rng.choice(NB, size=c, replace=False))
                if i == 4:
                    cols = np.array([NB - 1])
                idx[b, h, i, :c] = cols
                cnt[b, h, i] = len(cols)
    _run_sparse_case(w, 3, idx, cnt)


@pytest.mark.parametrize("step,expect_redo,heads", [(1.0, False, 4), (16.0, True, 4), (16.0, True, 12), (16.0, True, 20)])
def test_sparse_attention_row_maxima_growing_along_the_key_axis(step, expect_redo, heads):
    """Logits that grow from key block to key block.  The fast kernel keeps the first tile's row maximum
    as its reference: a moderate growth stays inside its headroom, a steep one makes it hand the work item
    to exact rescaling (listed behind the status record in the workspace).  Both must match the oracle; in the
    steep case items must actually have been handed over.  With 12 heads (6936 tile pairs, below 64 per SM) every
    CTA of the tile kernel recomputes several of its own, with 20 (11560) every CTA of the grid behind it does."""
    import dataclasses
    w = dataclasses.replace(wl.WORKLOADS["medium128"], H=heads)
    q, k, v = wl.make_self_qkv(w, 6)
    NB = w.n_blocks
    u = 1.0 / np.sqrt(w.d)
    q = (q.float() + 8.0 * u).to(torch.bfloat16)
    ramp = torch.arange(w.n_video, dtype=torch.float32).div(w.blk, rounding_mode="floor") * step
    k = (k.float() + (ramp * u).view(1, 1, -1, 1)).to(torch.bfloat16)
    rng = np.random.default_rng(8)
    idx = np.full((w.B, w.H, NB, NB), -1, np.int32)
    cnt = np.zeros((w.B, w.H, NB), np.int32)
    for b in range(w.B):
        for h in range(w.H):
            for i in range(NB):
                c = NB if i % 4 == 0 else 1 + int(rng.integers(NB))
                cols = np.sort(rng.choice(NB, size=c, replace=False))
                idx[b, h, i, :c] = cols
                cnt[b, h, i] = c
    o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(),
                                          torch.from_numpy(cnt).cuda(), w.blk, want_lse=True)
    _status_ok(ws)
    want_o, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, w.blk)
    _close(_np64(o), want_o, "growing maxima O")
    _close_lse(_np64(lse), want_l, "growing maxima lse")
    n_redo, items = av.avsa_sparse_self_attn_redo_items(ws)
    assert (n_redo > 0) == expect_redo
    if heads > 4:
        assert n_redo > 2 * 148
    if expect_redo:
        assert len(set(items.tolist())) == n_redo and items.min() >= 0 and items.max() < w.B * w.H * NB
        # items with a single key block never outgrow their reference
        assert np.all(cnt.reshape(-1)[items] > 1)


def test_sparse_attention_is_reproducible_over_repeated_launches():
    """Same inputs, 25 launches into fresh outputs: every result is bit-identical (the accumulation order is
    fixed by the lists, so any difference would be a race between the pipeline's stages)."""
    w = wl.WORKLOADS["medium128"]
    q, k, v = (t.cuda() for t in wl.make_self_qkv(w, 9))
    NB = w.n_blocks
    rng = np.random.default_rng(11)
    idx = np.full((w.B, w.H, NB, NB), -1, np.int32)
    cnt = np.zeros((w.B, w.H, NB), np.int32)
    for b in range(w.B):
        for h in range(w.H):
            for i in range(NB):
                c = 1 + int(rng.integers(NB))
                idx[b, h, i, :c] = np.sort(rng.choice(NB, size=c, replace=False))
                cnt[b, h, i] = c
    idx_d, cnt_d = torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()
    first, first_lse, ws = av.avsa_sparse_self_attn(q, k, v, idx_d, cnt_d, w.blk, want_lse=True)
    _status_ok(ws)
    for _ in range(24):
        o, lse, ws = av.avsa_sparse_self_attn(q, k, v, idx_d, cnt_d, w.blk, want_lse=True)
        assert torch.equal(o, first) and torch.equal(lse, first_lse)
    _status_ok(ws)
    want_o, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, w.blk)
    _close(_np64(first), want_o, "random lists O")
    _close_lse(_np64(first_lse), want_l, "random lists lse")


def test_sparse_attention_strided_bnhd_layout():
    w = wl.WORKLOADS["small128"]
    q, k, v = wl.make_self_qkv(w, 4)
    NB = w.n_blocks
    idx = np.broadcast_to(np.arange(NB, dtype=np.int32), (w.B, w.H, NB, NB)).copy()
    cnt = np.full((w.B, w.H, NB), NB, np.int32)
    # storage [B,N,H,d], viewed as [B,H,N,d]
    qs, ks, vs = (t.cuda().permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (q, k, v))
    assert not qs.is_contiguous()
    o, _, ws = av.avsa_sparse_self_attn(qs, ks, vs, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), w.blk)
    _status_ok(ws)
    assert o.stride() == qs.stride()
    want, _ = orc.dense_attention(_np64(q), _np64(k), _np64(v))
    _close(_np64(o), want, "strided O")


@pytest.mark.parametrize("seed", range(8))
def test_sparse_attention_random_shapes_and_lists(seed):
    """Seeded random shapes (batch, heads, length incl. ragged tails and lengths below one block, both tile
    sizes) with random ascending lists of random length, against the oracle."""
    rng = np.random.default_rng(100 + seed)
    d = int(rng.choice([64, 128]))
    blk = d
    B, H = int(rng.integers(1, 4)), int(rng.integers(1, 6))
    N = int(rng.integers(1, 9 * blk))
    NB = (N + blk - 1) // blk
    g = torch.Generator().manual_seed(200 + seed)
    q, k, v = (torch.randn(B, H, N, d, generator=g).to(torch.bfloat16) for _ in range(3))
    idx = np.full((B, H, NB, NB), -1, np.int32)
    cnt = np.zeros((B, H, NB), np.int32)
    for b in range(B):
        for h in range(H):
            for i in range(NB):
                c = 1 + int(rng.integers(NB))
                idx[b, h, i, :c] = np.sort(rng.choice(NB, size=c, replace=False))
                cnt[b, h, i] = c
    o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(),
                                          torch.from_numpy(cnt).cuda(), blk, want_lse=True)
    _status_ok(ws)
    assert av.avsa_redo_count(ws) == 0             # unit-variance logits: nothing outgrows its reference
    want_o, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, blk)
    _close(_np64(o), want_o, f"random shape B{B} H{H} N{N} d{d} O")
    _close_lse(_np64(lse), want_l, f"random shape B{B} H{H} N{N} d{d} lse")


def test_sparse_attention_rows_not_32_byte_aligned():
    """Rows 272 bytes apart (d padded by 8 elements): 16-byte aligned, which is all the interface asks for (the
    tile loads and the staged tile store go through tensor maps).  Same result as the contiguous layout, bit for bit."""
    w = wl.WORKLOADS["medium128"]
    q, k, v = wl.make_self_qkv(w, 12)
    NB = w.n_blocks
    _, _, _, s64 = _oracle_scores(w, 0)
    n_protect = orc.ceil_pct(w.protect_pct, w.n_video)
    k_keep = max(1, orc.ceil_pct(w.keep_pct, NB))
    _, _, idx, cnt, _, _ = _oracle_mask(w, q, k, s64, n_protect, k_keep)

    def padded(t):
        buf = torch.zeros(t.shape[:-1] + (w.d + 8,), dtype=t.dtype, device="cuda")
        buf[..., : w.d] = t.cuda()
        return buf[..., : w.d]

    qp, kp, vp = padded(q), padded(k), padded(v)
    assert qp.stride(2) == w.d + 8 and qp.stride(3) == 1
    o, lse, ws = av.avsa_sparse_self_attn(qp, kp, vp, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), w.blk,
                                          want_lse=True)
    _status_ok(ws)
    assert o.stride() == qp.stride()
    want_o, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, w.blk)
    _close(_np64(o), want_o, "padded rows O")
    _close_lse(_np64(lse), want_l, "padded rows lse")
    # and the contiguous layout gives the same numbers bit for bit
    o2, lse2, ws2 = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(),
                                             torch.from_numpy(cnt).cuda(), w.blk, want_lse=True)
    _status_ok(ws2)
    assert torch.equal(o2, o.contiguous()) and torch.equal(lse2, lse)


def test_sparse_attention_rejects_malformed_lists_without_touching_memory():
    w = wl.WORKLOADS["small128"]
    q, k, v = (t.cuda() for t in wl.make_self_qkv(w, 0))
    NB = w.n_blocks
    for bad in ([0, 0], [2, 1], [0, NB], [-1, 1]):
        idx = np.broadcast_to(np.arange(NB, dtype=np.int32), (w.B, w.H, NB, NB)).copy()
        cnt = np.full((w.B, w.H, NB), NB, np.int32)
        idx[0, 1, 2, :2] = bad
        cnt[0, 1, 2] = 2
        o, _, ws = av.avsa_sparse_self_attn(q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), w.blk)
        code, detail = av.avsa_read_status(ws)
        assert code == av.AVSA_ERR_BAD_MASK
        assert detail[1] == (0 * w.H + 1) * NB + 2
    cnt = np.zeros((w.B, w.H, NB), np.int32)
    o, _, ws = av.avsa_sparse_self_attn(q, k, v, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), w.blk)
    assert av.avsa_read_status(ws)[0] == av.AVSA_ERR_BAD_MASK


def test_sparse_attention_skips_only_the_malformed_item_of_a_long_queue():
    """408 work items on 148 persistent CTAs, three of them malformed (bad count, descending entries, entry out
    of range): the status says BAD_MASK, the malformed items' rows are left untouched, every other row is right."""
    import dataclasses
    w = dataclasses.replace(wl.WORKLOADS["medium128"], H=12)
    q, k, v = wl.make_self_qkv(w, 13)
    NB = w.n_blocks
    rng = np.random.default_rng(14)
    idx = np.full((w.B, w.H, NB, NB), -1, np.int32)
    cnt = np.zeros((w.B, w.H, NB), np.int32)
    for b in range(w.B):
        for h in range(w.H):
            for i in range(NB):
                c = 1 + int(rng.integers(6))
                idx[b, h, i, :c] = np.sort(rng.choice(NB, size=c, replace=False))
                cnt[b, h, i] = c
    good_idx, good_cnt = idx.copy(), cnt.copy()
    bad_items = [(0, 3, 5), (1, 7, 0), (1, 11, 16)]
    cnt[0, 3, 5] = NB + 1
    idx[1, 7, 0, :2] = [4, 2]; cnt[1, 7, 0] = 2
    idx[1, 11, 16, :1] = [NB]; cnt[1, 11, 16] = 1
    o = torch.full((w.B, w.H, w.n_video, w.d), 7.0, dtype=torch.bfloat16, device="cuda")
    _, _, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(),
                                        torch.from_numpy(cnt).cuda(), w.blk, o=o)
    code, detail = av.avsa_read_status(ws)
    assert code == av.AVSA_ERR_BAD_MASK
    assert detail[1] in [(b * w.H + h) * NB + i for b, h, i in bad_items]
    want, _ = orc.masked_attention(_np64(q), _np64(k), _np64(v), good_idx, good_cnt, w.blk)
    got = _np64(o)
    for b, h, i in bad_items:
        lo, hi = i * w.blk, min((i + 1) * w.blk, w.n_video)
        assert np.all(got[b, h, lo:hi] == 7.0)              # refused: nothing written
        want[b, h, lo:hi] = 7.0
    _close(got, want, "queue with malformed items")


@pytest.mark.parametrize("heads", [2, 6])
@pytest.mark.parametrize("bad", [None, 35])
def test_sparse_attention_list_lengths(heads, bad):
    """Lists around the 32 entries that are read at once, and an entry behind them that is out of order; with an item per CTA at
    most (2 heads x 66 query blocks, the output staged over Q) and off the queue."""
    B, N, d = 1, 64 * 65 + 9, 64
    NB = 66
    g = torch.Generator().manual_seed(heads)
    q, k, v = (torch.randn((B, heads, N, d), generator=g).to(torch.bfloat16) for _ in range(3))
    rng = np.random.default_rng(3)
    idx = np.full((B, heads, NB, NB), -1, np.int32)
    cnt = np.zeros((B, heads, NB), np.int32)
    for h in range(heads):
        for i in range(NB):
            c = [1, 2, 3, 31, 32, 33, 63, 64, 65, 66][(h + i) % 10]
            idx[0, h, i, :c] = np.sort(rng.choice(NB, size=c, replace=False))
            cnt[0, h, i] = c
    want, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, d)
    if bad is not None:
        assert cnt[0, 1, 5] == 63
        idx[0, 1, 5, bad] = idx[0, 1, 5, bad - 1]
        want[0, 1, 5 * d : 6 * d] = 7.0
    o = torch.full((B, heads, N, d), 7.0, dtype=torch.bfloat16, device="cuda")
    _, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(),
                                          d, want_lse=True, o=o)
    code, detail = av.avsa_read_status(ws)
    if bad is None:
        assert code == av.AVSA_OK
        _close_lse(_np64(lse), want_l, "list lengths lse")
    else:
        assert code == av.AVSA_ERR_BAD_MASK and detail[1] == NB + 5
    _close(_np64(o), want, "list lengths O")


@pytest.mark.parametrize("case", ["random", "nothing_shared", "first_blocks_swapped", "dense_beside_short", "outgrown", "nan_value",
                                  "both_malformed", "window"])
def test_sparse_attention_pairs_of_64_blocks(case):
    """Query blocks of 64 rows are taken two at a time with the union of their lists: an odd number of blocks (the last pair has one
    block, of 9 rows), lists that share nothing or begin elsewhere, a block that one of a pair does not list and whose values are no
    numbers, rows that outgrow their reference in one block of a pair, a pair without a list, and more than the 1024 key blocks that
    are joined at a time."""
    B, H, NB, d = (1, 1, 1061, 64) if case == "window" else (1, 17, 35, 64)
    N = (NB - 1) * d + 9
    g = torch.Generator().manual_seed(3)
    q, k, v = (torch.randn((B, H, N, d), generator=g).to(torch.bfloat16) for _ in range(3))
    rng = np.random.default_rng(11)
    idx = np.full((B, H, NB, NB), -1, np.int32)
    cnt = np.zeros((B, H, NB), np.int32)
    for h in range(H):
        for i in range(NB):
            cols = rng.choice(NB, size=1 + int(rng.integers(6)) if case == "window" else 1 + int(rng.integers(NB)), replace=False)
            if case == "window":
                cols = np.union1d(cols, [[0, 1023, 1024], [1024], [1060], [1023]][i % 4])
            elif case == "nothing_shared":
                cols = np.arange(i % 2, NB, 2 + i % 3 * 2)
            elif case == "first_blocks_swapped":
                cols = np.arange(7 + i % 5 if i % 4 in (0, 3) else i % 5, NB)
            elif case == "dense_beside_short":
                cols = np.arange(NB) if (i // 2) % 2 == i % 2 else np.array([(5 * i) % NB])
            elif case == "nan_value":
                cols = np.union1d(cols[cols != 7], [0] if i != 8 else [7])
            cols = np.sort(cols)
            idx[0, h, i, : len(cols)], cnt[0, h, i] = cols, len(cols)
    if case == "outgrown":      # keys that grow from block to block, for the rows of every other block of a pair
        q[:, :, (torch.arange(N) // d) % 2 == 1] *= 0.01
        k = (k.float() * (1 + 3 * (torch.arange(N) // d))[None, None, :, None]).to(torch.bfloat16)
    want, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, d)
    if case == "nan_value":
        v[:, :, 7 * d : 8 * d] = float("nan")
        want[:, :, 8 * d : 9 * d] = 7.0
    if case == "both_malformed":
        cnt[0, 2, 10], cnt[0, 2, 11] = 0, NB + 1
        want[0, 2, 10 * d : 12 * d] = want_l[0, 2, 10 * d : 12 * d] = 7.0
    o = torch.full((B, H, N, d), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H, N), 7.0, device="cuda")
    _, _, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), d,
                                        want_lse=True, o=o, lse=lse)
    code, detail = av.avsa_read_status(ws)
    if case == "both_malformed":
        assert code == av.AVSA_ERR_BAD_MASK and detail[1] in (2 * NB + 10, 2 * NB + 11)
    else:
        assert code == av.AVSA_OK
    got = _np64(o)
    n_redo, items = av.avsa_sparse_self_attn_redo_items(ws)
    if case == "nan_value":
        assert np.all(np.isnan(got[:, :, 8 * d : 9 * d]))      # these rows list the block
        got[:, :, 8 * d : 9 * d] = 7.0
    elif case == "outgrown":
        assert n_redo > 0 and len(set(items.tolist())) == n_redo and np.all(cnt.reshape(-1)[items] > 1)
        assert np.all(items % NB % 2 == 0)
    else:
        assert n_redo == 0
    _close(got, want, f"pairs {case} O")
    _close_lse(_np64(lse), want_l, f"pairs {case} lse")


def _random_lists(rng, B, H, NB, longest):
    idx, cnt = np.full((B, H, NB, NB), -1, np.int32), np.zeros((B, H, NB), np.int32)
    for at in np.ndindex(B, H, NB):
        c = NB if rng.integers(12) == 0 and longest > 8 else 1 + int(rng.integers(longest))
        idx[at][:c], cnt[at] = np.sort(rng.choice(NB, size=c, replace=False)), c
    return idx, cnt


def _runs_in_pairs(B, H, N):
    """The workspace has room for the joint lists of two query blocks each."""
    NB, up = (N + 63) // 64, lambda x: (x + 255) // 256 * 256
    NP = (NB + 1) // 2
    return av.avsa_sparse_self_attn_workspace_bytes(B, H, N, 64, 64) == 256 + up(B * H * NB * 8) + up(B * H * NP * (2 * NP + 1) * 4)


@pytest.mark.parametrize("layout", ["bhnd", "bnhd", "padded"])
def test_sparse_attention_pairs_in_batches_layouts_and_used_buffers(layout):
    """Two batch items with lists of their own and an odd number of blocks, read through strides: the same bits as from contiguous tensors,
    whatever workspace and outputs held before, launch by launch, and from a CUDA graph."""
    B, H, NB, d = 2, 2, 67, 64
    N = (NB - 1) * d + 9
    assert _runs_in_pairs(B, H, N)
    g = torch.Generator().manual_seed(8)
    cpu = [torch.randn((B, H, N, d), generator=g).to(torch.bfloat16) for _ in range(3)]
    idx, cnt = _random_lists(np.random.default_rng(5), B, H, NB, NB // 2)
    idx_d, cnt_d = torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()
    want_o, want_lse, ws = av.avsa_sparse_self_attn(*(t.cuda() for t in cpu), idx_d, cnt_d, d, want_lse=True)
    _status_ok(ws)
    if layout == "bhnd":
        ref_o, ref_lse = orc.masked_attention(*(_np64(t) for t in cpu), idx, cnt, d)
        _close(_np64(want_o), ref_o, "pairs of two batch items O")
        _close_lse(_np64(want_lse), ref_lse, "pairs of two batch items lse")

    def store(t):
        if layout == "bnhd":
            return t.cuda().transpose(1, 2).contiguous().transpose(1, 2)
        buf = torch.zeros(t.shape[:-1] + (d + (8 if layout == "padded" else 0),), dtype=t.dtype, device="cuda")
        buf[..., :d] = t.cuda()
        return buf[..., :d]
    q, k, v = (store(t) for t in cpu)
    n = av.avsa_sparse_self_attn_workspace_bytes(B, H, N, d, d)
    for fill in (0x00, 0xFF):
        ws = torch.full((n,), fill, dtype=torch.uint8, device="cuda")
        o, lse = torch.empty_strided(q.shape, q.stride(), dtype=torch.bfloat16, device="cuda"), torch.empty((B, H, N), device="cuda")
        for _ in range(3):
            o.fill_(float(fill))
            lse.fill_(float(fill))
            av.avsa_sparse_self_attn(q, k, v, idx_d, cnt_d, d, o=o, lse=lse, ws=ws)
            _status_ok(ws)
            assert torch.equal(o, want_o) and torch.equal(lse, want_lse)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        av.avsa_sparse_self_attn(q, k, v, idx_d, cnt_d, d, o=o, lse=lse, ws=ws)
    for _ in range(2):
        o.zero_()
        lse.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(o, want_o) and torch.equal(lse, want_lse)


def test_sparse_attention_pairs_whose_blocks_both_outgrow_their_reference():
    """Keys that grow from block to block for every row, in two batch items: both blocks of a pair are recomputed, each with its list."""
    B, H, NB, d = 2, 3, 65, 64
    N = NB * d
    assert _runs_in_pairs(B, H, N)
    g = torch.Generator().manual_seed(6)
    q, k, v = (torch.randn((B, H, N, d), generator=g) for _ in range(3))
    k[:, 1:] *= (1 + 3 * (torch.arange(N) // d))[None, None, :, None]      # (the first head's keys do not grow)
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    idx, cnt = _random_lists(np.random.default_rng(9), B, H, NB, 12)
    o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), d, want_lse=True)
    _status_ok(ws)
    n_redo, items = av.avsa_sparse_self_attn_redo_items(ws)
    assert n_redo > 0 and len(set(items.tolist())) == n_redo and np.all(cnt.reshape(-1)[items] > 1)
    b, h, block = items // (H * NB), items // NB % H, items % NB
    assert np.all(h > 0) and set(b.tolist()) == {0, 1}
    assert len({(x, y, z // 2) for x, y, z in zip(b, h, block)}) < n_redo      # both of a pair, somewhere
    want, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, d)
    _close(_np64(o), want, "pairs recomputed O")
    _close_lse(_np64(lse), want_l, "pairs recomputed lse")


@pytest.mark.parametrize("b,h,block,bad", [(1, 1, 66, "empty"), (1, 0, 5, "order"), (1, 1, 4, "range"), (0, 1, 7, "long")])
def test_sparse_attention_pairs_with_a_malformed_list_in_either_batch_item(b, h, block, bad):
    """The item that is reported is the query block's, its rows stay as they were, and its neighbour in the pair has its own list."""
    B, H, NB, d = 2, 2, 67, 64
    N = (NB - 1) * d + 9
    assert _runs_in_pairs(B, H, N)
    g = torch.Generator().manual_seed(7)
    q, k, v = (torch.randn((B, H, N, d), generator=g).to(torch.bfloat16) for _ in range(3))
    idx, cnt = _random_lists(np.random.default_rng(3), B, H, NB, 7)
    want, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, d)
    row = idx[b, h, block]
    if bad == "order":
        row[:2], cnt[b, h, block] = (9, 9), 2
    elif bad == "range":
        row[0], cnt[b, h, block] = NB, 1
    else:
        cnt[b, h, block] = 0 if bad == "empty" else NB + 1
    want[b, h, block * d:(block + 1) * d] = want_l[b, h, block * d:(block + 1) * d] = 7.0
    o, lse = torch.full((B, H, N, d), 7.0, dtype=torch.bfloat16, device="cuda"), torch.full((B, H, N), 7.0, device="cuda")
    _, _, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), d, o=o, lse=lse)
    code, detail = av.avsa_read_status(ws)
    assert code == av.AVSA_ERR_BAD_MASK and detail[1:] == ((b * H + h) * NB + block, cnt[b, h, block])
    _close(_np64(o), want, f"pairs, {bad} list O")
    _close_lse(_np64(lse), want_l, f"pairs, {bad} list lse")


@pytest.mark.parametrize("flags", [av.AVSA_PROTECT_ROWS, av.AVSA_PROTECT_ROWS | av.AVSA_PROTECT_COLS])
def test_sparse_attention_pairs_under_the_masks_own_lists(flags):
    """Mask and attention of 64-blocks with protected rows, and protected columns too."""
    B, H, N, d = 2, 4, 70 * 64 + 9, 64
    assert _runs_in_pairs(B, H, N)
    g = torch.Generator().manual_seed(2)
    q, k, v = (torch.randn((B, H, N, d), generator=g).to(torch.bfloat16) for _ in range(3))
    s = torch.rand((B, N), generator=g)
    s[:, 1000:1400] += 1.0
    m = av.avsa_build_block_mask(q.cuda(), k.cuda(), s.cuda(), 300, 7, d, flags=flags)
    _status_ok(m["ws"])
    o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), m["col_idx"], m["col_cnt"], d, want_lse=True)
    _status_ok(ws)
    want, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), m["col_idx"].cpu().numpy(), m["col_cnt"].cpu().numpy(), d)
    _close(_np64(o), want, "pairs under a mask O")
    _close_lse(_np64(lse), want_l, "pairs under a mask lse")


def test_sparse_attention_pairs_of_more_than_two_windows_of_blocks():
    """Lists are joined 1024 key blocks at a time: three windows, entries at their edges, the last pair a single block."""
    B, H, NB, d = 1, 1, 2101, 64
    N = (NB - 1) * d + 33
    assert _runs_in_pairs(B, H, N)
    g = torch.Generator().manual_seed(1)
    q, k, v = (torch.randn((B, H, N, d), generator=g).to(torch.bfloat16) for _ in range(3))
    rng = np.random.default_rng(4)
    idx, cnt = np.full((B, H, NB, NB), -1, np.int32), np.zeros((B, H, NB), np.int32)
    for i in range(NB):
        cols = np.union1d(rng.choice(NB, size=int(rng.integers(1, 4))), [[0, 1023, 1024], [2047, 2048], [1024, 2100], [2048], []][i % 5]).astype(np.int32)
        idx[0, 0, i, :len(cols)], cnt[0, 0, i] = cols, len(cols)
    o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), d, want_lse=True)
    _status_ok(ws)
    want, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, d)
    _close(_np64(o), want, "three windows O")
    _close_lse(_np64(lse), want_l, "three windows lse")


# ------------------------------------------------------------------------------------------- cross attention
@pytest.mark.parametrize("name", ["tiny", "small128", "medium128"])
def test_cross_attention_outputs_and_scores(name):
    w = wl.WORKLOADS[name]
    (qa, kc, vc), want_o, want_lse, want_s = _oracle_scores(w, 0)
    gamma = 1.0 / (w.H * w.n_audio)
    o, lse, s, ws = av.avsa_cross_attn_scores(qa.cuda(), kc.cuda(), vc.cuda(), score_gamma=gamma)
    _status_ok(ws)
    assert av.avsa_redo_count(ws) == 0             # the planted boost (a few nats) stays inside the fast kernel's range
    _close(_np64(o), want_o, f"{name} cross O")
    _close_lse(_np64(lse), want_lse, f"{name} cross lse")
    got_s = _np64(s)
    assert abs(got_s.sum() - w.B) < 2e-3 * w.B                          # rows of Eq. 1 sum to one
    _close_scores(got_s, want_s, f"{name} scores (L1 norm)")
    # raw column mass (gamma = 1): every video token's score on its own, so that a wrong column cannot hide
    _, _, s_raw, _ = av.avsa_cross_attn_scores(qa.cuda(), kc.cuda(), vc.cuda(), score_gamma=1.0, want_o=False)
    _close_scores(_np64(s_raw), want_s * (w.H * w.n_audio), f"{name} scores (raw column mass)")
    # running blend (Eq. 4) and bit-for-bit reproducibility
    prev = torch.rand_like(s) * float(want_s.max())
    s2 = prev.clone()
    av.avsa_cross_attn_scores(qa.cuda(), kc.cuda(), vc.cuda(), scores=s2, score_beta=0.25, score_gamma=0.75 * gamma)
    torch.cuda.synchronize()
    want2 = 0.25 * _np64(prev) + 0.75 * want_s
    _close_scores(_np64(s2), want2, f"{name} blended scores (Eq. 4)")
    _, _, s3, _ = av.avsa_cross_attn_scores(qa.cuda(), kc.cuda(), vc.cuda(), score_gamma=gamma)
    assert torch.equal(s, s3)


def test_cross_attention_long_query_axis_in_chunks():
    """More than 256 queries: the column-sum pass splits the query axis in four."""
    w = wl.Workload("x", 1, 2, 128, 2, 9, 17, 300, 128, 50, 10, 1.0, ((0, 1, 1, 3, 2, 4),))
    (qa, kc, vc), want_o, want_lse, want_s = _oracle_scores(w, 7)
    o, lse, s, ws = av.avsa_cross_attn_scores(qa.cuda(), kc.cuda(), vc.cuda(), score_gamma=1.0 / (w.H * w.n_audio))
    _status_ok(ws)
    _close(_np64(o), want_o, "cross O")
    _close_lse(_np64(lse), want_lse, "cross lse")
    _close_scores(_np64(s), want_s, "scores, four query chunks")


@pytest.mark.parametrize("B,H,Nq,Nk,d,scores", [
    (1, 1, 1, 1, 128, True),           # one query, one key
    (1, 1, 600, 3000, 128, False),     # 5 query tiles in chunks of 4, 24 key tiles cut into twelve ranges
    (1, 2, 300, 2900, 128, True),      # 3 query tiles, split rows, the LSEs of the score pass from the parts
    (2, 3, 140, 333, 64, True),        # few tiles: whole rows, written by the tile kernel itself
    (1, 22, 2427, 200, 128, True),     # few keys: both passes in one kernel, 418 query tiles over the CTAs
    (1, 22, 2427, 300, 128, True),     # reverse: 19 query tiles, score pass with three key tiles resident
    (1, 22, 2427, 300, 64, True),
    (2, 2, 600, 257, 64, True),        # reverse with one key in the last tile
    (2, 2, 600, 257, 128, True),
    (1, 4, 700, 385, 128, True),
    (1, 2, 513, 512, 64, True),        # the fewest queries and the most keys of the reverse direction
    (1, 3, 1000, 512, 128, True),
    (1, 2, 130, 6400, 64, True),
    (1, 100, 40, 1000, 64, True),      # score pass: 800 key tiles cut evenly through the heads
    (1, 96, 300, 520, 128, True),      # the same with the queries in four chunks
    (1, 3, 128, 700, 64, True),        # one chunk, tiles by turns over two groups
    (1, 3, 129, 650, 128, True),       # one chunk of 144
    (1, 2, 256, 515, 128, True),
    (1, 2, 257, 900, 64, True),        # four chunks of 80
    (2, 2, 512, 640, 128, True),
    (1, 1, 100, 6400, 64, True),       # a row in more parts than lanes take at once (50 of 16 and, below, of 32)
    (1, 1, 130, 6400, 128, True),
    (1, 1, 100, 17000, 64, True),      # more parts (133 and, with as many as there are SMs, 148) than the merge's table of weights holds
    (1, 1, 100, 18900, 128, True),
    (1, 40, 400, 900, 64, True),       # more than 8192 split rows
    (1, 20, 500, 1700, 128, True),
])
def test_cross_attention_work_split(B, H, Nq, Nk, d, scores):
    """The ways a stream of (query tile, key tile) pairs is cut over the CTAs: whole rows, split rows, chunks that do not divide
    the query tiles; with O, and with only the LSE asked for (same LSEs)."""
    g = torch.Generator().manual_seed(Nq * 7 + Nk)
    q, k, v = (torch.randn((B, H, n, d), generator=g).to(torch.bfloat16) for n in (Nq, Nk, Nk))
    want_o, want_lse, A = orc.cross_attention(_np64(q), _np64(k), _np64(v))
    o, lse, s, ws = av.avsa_cross_attn_scores(q.cuda(), k.cuda(), v.cuda(), want_scores=scores, score_gamma=1.0 / (H * Nq))
    _status_ok(ws)
    _close(_np64(o), want_o, "split O")
    _close_lse(_np64(lse), want_lse, "split lse")
    if scores:
        _close_scores(_np64(s), orc.column_scores(A, gamma=1.0 / (H * Nq)), "split scores")
    _, lse2, _, ws2 = av.avsa_cross_attn_scores(q.cuda(), k.cuda(), v.cuda(), want_scores=False, want_o=False)
    _status_ok(ws2)
    assert torch.equal(lse, lse2)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,Nq,Nk", [
    (1, 1, 1, 32), (1, 2, 127, 33), (2, 3, 1000, 64), (1, 40, 600, 65), (1, 40, 515, 100), (1, 24, 2427, 128),
    (1, 3, 129, 129), (1, 40, 600, 160), (2, 20, 515, 161), (1, 24, 2427, 200), (1, 2, 128, 255), (1, 40, 600, 256),
])
def test_cross_attention_few_keys(B, H, Nq, Nk, d):
    """K and V of a head on chip, both passes in one kernel: one and two key groups, chunks of 32 keys and their remainders, one
    and several query tiles and heads per CTA; the same bits without scores and on a second run."""
    g = torch.Generator().manual_seed(Nq * 7 + Nk)
    q, k, v = (torch.randn((B, H, n, d), generator=g).to(torch.bfloat16) for n in (Nq, Nk, Nk))
    hs = sorted({0, H // 2, H - 1})
    gamma = 1.0 / (H * Nq)
    qc, kc, vc = (t.transpose(1, 2).contiguous().transpose(1, 2).cuda() for t in (q, k, v))
    o, lse, s, ws = av.avsa_cross_attn_scores(qc, kc, vc, score_gamma=gamma)
    _status_ok(ws)
    assert av.avsa_redo_count(ws) == 0
    want_s = np.zeros((B, Nk))
    for h in range(H):
        want_o, want_lse, A = orc.cross_attention(_np64(q[:, h : h + 1]), _np64(k[:, h : h + 1]), _np64(v[:, h : h + 1]))
        want_s = orc.column_scores(A, s_prev=want_s, beta=1.0, gamma=gamma)
        if h in hs:
            _close(_np64(o[:, h : h + 1]), want_o, "few keys O")
            _close_lse(_np64(lse[:, h : h + 1]), want_lse, "few keys lse")
    _close_scores(_np64(s), want_s, "few keys scores")
    o2, lse2, _, ws2 = av.avsa_cross_attn_scores(qc, kc, vc, want_scores=False)
    _status_ok(ws2)
    assert torch.equal(o, o2) and torch.equal(lse, lse2)
    s3 = av.avsa_cross_attn_scores(qc, kc, vc, want_o=False, score_gamma=gamma)[2]
    assert torch.equal(s, s3)


@pytest.mark.parametrize("step", [30.0, 80.0])
def test_cross_attention_few_keys_that_outgrow_their_reference(step):
    """The keys from 128 on have logits larger by 30 nats (43 in base 2, up to 62 in some rows: not counted, and most rows stay
    relative to the first ones' maximum) or 80 (115: the rows take another reference, and their tiles are counted)."""
    B, H, Nq, Nk, d = 1, 3, 300, 200, 128
    g = torch.Generator().manual_seed(9)
    q, k, v = (torch.randn((B, H, n, d), generator=g) for n in (Nq, Nk, Nk))
    u = 1.0 / np.sqrt(d)
    q = (q + 8.0 * u).to(torch.bfloat16)
    q[:, :, ::2] = (q[:, :, ::2].float() - 8.0 * u).to(torch.bfloat16)      # every other row keeps its reference
    k[:, :, 128:] += step * u * np.sqrt(d) / 8.0
    k, v = k.to(torch.bfloat16), v.to(torch.bfloat16)
    o, lse, s, ws = av.avsa_cross_attn_scores(q.cuda(), k.cuda(), v.cuda(), score_gamma=1.0 / (H * Nq))
    _status_ok(ws)
    assert av.avsa_redo_count(ws) == (9 if step > 64 else 0)      # three tiles a head
    want_o, want_lse, A = orc.cross_attention(_np64(q), _np64(k), _np64(v))
    _close(_np64(o), want_o, "outgrown O")
    _close_lse(_np64(lse), want_lse, "outgrown lse")
    _close_scores(_np64(s), orc.column_scores(A, gamma=1.0 / (H * Nq)), "outgrown scores")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("nk", [200, 256])
@pytest.mark.parametrize("gap,v_first,v_rest", [(50, 59, 59), (63, 59, 59), (66, 59, 59), (61, 59, 0), (66, 59, 0), (200, 0, 59)])
def test_cross_attention_few_keys_with_large_values(gap, v_first, v_rest, nk, d):
    """The keys from 128 on have logits larger by ``gap`` in base 2 (within 2), and the values of either half are of magnitude 2^v:
    no accumulator overflows, and the first half keeps its weight where large values make it count (128 2^(59 - 61) beside
    72).  The tiles with a gap beyond 64 are counted."""
    B, H, Nq = 1, 2, 150
    g = torch.Generator().manual_seed(11)
    q, k, v = (torch.randn((B, H, n, d), generator=g) for n in (Nq, nk, nk))
    q, k = 0.5 * q, 0.5 * k
    q[..., 0], k[..., 0] = 8.0, 0.0
    k[:, :, 128:, 0] = gap / 8.0 * np.log(2.0) * np.sqrt(d)
    v = 1.0 + 0.25 * v
    v[:, :, :128] *= 2.0**v_first
    v[:, :, 128:] *= 2.0**v_rest
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    want_o, want_lse, A = orc.cross_attention(_np64(q), _np64(k), _np64(v))
    o, lse, s, ws = av.avsa_cross_attn_scores(q.cuda(), k.cuda(), v.cuda(), score_gamma=1.0 / (H * Nq))
    _status_ok(ws)
    assert av.avsa_redo_count(ws) == (2 * H if gap > 64 else 0)
    _close(_np64(o) / 2.0**v_rest, want_o / 2.0**v_rest, "large values O")
    _close_lse(_np64(lse), want_lse, "large values lse")
    _close_scores(_np64(s), orc.column_scores(A, gamma=1.0 / (H * Nq)), "large values scores")


@pytest.mark.parametrize("name", ["tiny", "small128", "medium128"])
def test_cross_attention_reverse_direction(name):
    """Video queries attending to audio keys (the other half of the bidirectional pair): outputs, LSE, and the
    audio-token saliency as column sums over the video queries (handled "analogously", Sec. 4.1)."""
    w = wl.WORKLOADS[name]
    qa, kc, vc = wl.make_cross_qkv(w, 3)
    q_video, k_audio, v_audio = kc, qa, wl.make_cross_qkv(w, 4)[0]          # roles swapped; fresh audio values
    want_o, want_lse, A = orc.cross_attention(_np64(q_video), _np64(k_audio), _np64(v_audio))
    gamma = 1.0 / (w.H * w.n_video)
    want_s = orc.column_scores(A, gamma=gamma)
    o, lse, s, ws = av.avsa_cross_attn_scores(q_video.cuda(), k_audio.cuda(), v_audio.cuda(), score_gamma=gamma)
    _status_ok(ws)
    _close(_np64(o), want_o, f"{name} reverse O")
    _close_lse(_np64(lse), want_lse, f"{name} reverse lse")
    got_s = _np64(s)
    assert got_s.shape == (w.B, w.n_audio)
    assert abs(got_s.sum() - w.B) < 2e-3 * w.B
    _close_scores(got_s, want_s, f"{name} reverse scores")
    _, _, s2, _ = av.avsa_cross_attn_scores(q_video.cuda(), k_audio.cuda(), v_audio.cuda(), score_gamma=gamma)
    assert torch.equal(s, s2)                                              # fixed summation order


@pytest.mark.parametrize("B,H,Nq,Nk,d", [
    (1, 2, 72, 257, 128), (1, 3, 1, 288, 64), (1, 2, 127, 289, 128), (1, 72, 20, 512, 64), (1, 73, 20, 512, 64),      # two slices
    (1, 33, 60, 400, 128), (2, 3, 129, 513, 128), (1, 8, 512, 769, 64), (1, 24, 33, 1280, 128), (2, 5, 200, 1537, 64),
    (1, 14, 128, 2048, 128), (1, 20, 128, 2048, 128), (1, 3, 300, 2047, 64), (2, 4, 72, 2070, 128), (1, 2, 100, 4096, 64),
    (1, 3, 40, 4003, 128), (1, 2, 100, 4097, 128), (1, 24, 157, 400, 128), (1, 36, 128, 400, 128), (1, 37, 128, 400, 128)])
@pytest.mark.parametrize("growth", [0.0, 30.0, 90.0])
def test_cross_attention_sliced_keys(B, H, Nq, Nk, d, growth):
    """Short calls against 257 to 4096 keys: a cluster of CTAs takes a query tile, each some of the keys.  Slices of four chunks of 32 keys
    and of eight, the last key alone in its chunk, several query tiles, the limits of that way and the first length beyond
    (test_which_short_cross_attention_calls_slice_their_keys says which calls go it); logits that grow along the keys (base 2, per
    128 keys), so that the reference changes inside a slice and from slice to slice; [B,N,H,d] storage; with and without scores."""
    g = torch.Generator().manual_seed(Nk + Nq)
    q, k, v = (torch.randn((B, H, n, d), generator=g) for n in (Nq, Nk, Nk))
    if growth:
        u = 1.0 / np.sqrt(d)
        q = q * 0.1 + 8.0 * u
        ramp = torch.arange(Nk, dtype=torch.float32).div(128, rounding_mode="floor") * growth * np.log(2) * np.sqrt(d) / 8.0
        k = k + (ramp * u).view(1, 1, -1, 1)
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    want_o, want_lse, A = orc.cross_attention(_np64(q), _np64(k), _np64(v))
    qs, ks, vs = (t.cuda().transpose(1, 2).contiguous().transpose(1, 2) for t in (q, k, v))
    prev = torch.rand((B, Nk), generator=g).cuda()
    o, lse, s, ws = av.avsa_cross_attn_scores(qs, ks, vs, scores=prev.clone(), score_beta=0.5, score_gamma=0.5 / (H * Nq))
    _status_ok(ws)
    assert o.stride() == qs.stride()
    _close(_np64(o), want_o, "sliced O")
    _close_lse(_np64(lse), want_lse, "sliced lse")
    _close_scores(_np64(s), 0.5 * _np64(prev) + orc.column_scores(A, gamma=0.5 / (H * Nq)), "sliced scores")
    again = av.avsa_cross_attn_scores(qs, ks, vs, scores=prev.clone(), score_beta=0.5, score_gamma=0.5 / (H * Nq))
    assert torch.equal(again[0], o) and torch.equal(again[1], lse) and torch.equal(again[2], s)
    o2, lse2, _, ws2 = av.avsa_cross_attn_scores(qs, ks, vs, want_scores=False)
    _status_ok(ws2)
    _close(_np64(o2), want_o, "sliced O without scores")
    _close_lse(_np64(lse2), want_lse, "sliced lse without scores")
    assert torch.equal(o2, o) and torch.equal(lse2, lse)


@pytest.mark.parametrize("Nq,Nk,d", [(40, 333, 64), (40, 400, 128), (130, 700, 64), (72, 2048, 128)])
@pytest.mark.parametrize("first,last", [(0, 128), (128, 256), (224, 333), (0, 332)])
def test_cross_attention_sliced_keys_that_all_have_logits_of_minus_infinity(Nq, Nk, d, first, last):
    """Keys that mask themselves (products below the range of fp32) fill a half of a slice, a slice, or all but a few keys: they weigh
    nothing, and the rest of the row is as without them."""
    B, H = 1, 3
    g = torch.Generator().manual_seed(Nk)
    q, k, v = (torch.randn((B, H, n, d), generator=g) for n in (Nq, Nk, Nk))
    q = q.abs() + 0.1
    k[:, :, first:last] = -3e38
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    want_o, want_lse, A = orc.cross_attention(_np64(q), _np64(k), _np64(v))
    o, lse, s, ws = av.avsa_cross_attn_scores(q.cuda(), k.cuda(), v.cuda(), score_gamma=1.0 / (H * Nq))
    _status_ok(ws)
    _close(_np64(o), want_o, "masked keys O")
    _close_lse(_np64(lse), want_lse, "masked keys lse")
    _close_scores(_np64(s), orc.column_scores(A, gamma=1.0 / (H * Nq)), "masked keys scores")


def _went_sliced(B, H, Nq, Nk, d, **kw):
    """Runs a call of this shape on random tensors and tells by its workspace whether a cluster took each query tile: then a record per
    CTA begins behind the status record, all zeros where nothing went wrong."""
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v = (torch.randn((B, H, n, d), generator=g, device="cuda").bfloat16() for n in (Nq, Nk, Nk))
    ws = torch.full((av.avsa_cross_attn_scores_workspace_bytes(B, H, Nq, Nk, d),), 0xFF, dtype=torch.uint8, device="cuda")
    av.avsa_cross_attn_scores(q, k, v, ws=ws, **kw)
    _status_ok(ws)
    ctas = B * H * ((Nq + 127) // 128) * ((Nk + 255) // 256)
    return bool((ws[256:256 + 32 * ctas] == 0).all())


@pytest.mark.parametrize("B,H,Nq,Nk,d,sliced", [
    (1, 2, 72, 257, 128, True), (1, 3, 1, 288, 64, True), (1, 16, 128, 257, 128, True), (1, 17, 128, 257, 128, False), (1, 49, 128, 257, 64, False),
    (1, 32, 128, 300, 128, True), (1, 33, 128, 300, 128, False), (1, 36, 128, 400, 128, True), (1, 37, 128, 400, 128, False), (1, 24, 157, 400, 128, True),
    (1, 72, 20, 512, 64, True), (1, 36, 128, 640, 128, True), (1, 37, 128, 640, 128, False), (1, 24, 33, 1280, 128, True), (2, 4, 72, 2070, 128, True),
    (1, 2, 100, 4096, 64, True), (1, 2, 100, 4097, 128, False), (1, 2, 513, 400, 128, False), (1, 80, 20, 512, 64, False), (1, 20, 128, 2048, 128, False)])
def test_which_short_cross_attention_calls_slice_their_keys(B, H, Nq, Nk, d, sliced):
    """The limits of the sliced way on both sides, and its parity shapes: the tests that mean it reach it."""
    assert _went_sliced(B, H, Nq, Nk, d) == sliced
    assert _went_sliced(B, H, Nq, Nk, d, want_scores=False) == sliced


@pytest.mark.parametrize("Nk,d", [(1100, 64), (2048, 128), (4000, 128)])
def test_cross_attention_with_as_many_clusters_as_run_and_one_more(Nk, d):
    """The last number of query tiles that the device's clusters hold side by side, and the next: both against the oracle."""
    slices = (Nk + 255) // 256
    heads = next(h for h in range(1, 148 // slices + 2) if not _went_sliced(1, h, 128, Nk, d)) - 1
    assert heads >= 148 // slices // 2
    for H in (heads, heads + 1):
        g = torch.Generator().manual_seed(H)
        q, k, v = (torch.randn((1, H, n, d), generator=g).to(torch.bfloat16) for n in (128, Nk, Nk))
        o, lse, s, ws = av.avsa_cross_attn_scores(q.cuda(), k.cuda(), v.cuda(), score_gamma=1.0 / (H * 128))
        _status_ok(ws)
        want_o, want_lse, A = orc.cross_attention(_np64(q), _np64(k), _np64(v))
        _close(_np64(o), want_o, "clusters O")
        _close_lse(_np64(lse), want_lse, "clusters lse")
        _close_scores(_np64(s), orc.column_scores(A, gamma=1.0 / (H * 128)), "clusters scores")


@pytest.mark.parametrize("B,H,Nq,Nk,d", [
    (1, 24, 157, 400, 128), (1, 74, 55, 512, 128), (1, 74, 128, 512, 128), (1, 20, 128, 257, 128), (1, 44, 128, 640, 128), (1, 60, 128, 257, 64),
    (2, 4, 200, 1500, 64), (2, 3, 700, 100, 64), (1, 5, 700, 200, 128), (1, 4, 160, 6000, 128), (1, 6, 900, 300, 64)])
def test_cross_attention_gives_the_same_rows_with_scores_and_without(B, H, Nq, Nk, d):
    """The way a shape is computed does not depend on whether the response scores are wanted: sliced keys and the limits of that way, few
    keys, two passes, the reverse direction."""
    g = torch.Generator(device="cuda").manual_seed(Nk + Nq)
    q, k, v = (torch.randn((B, H, n, d), generator=g, device="cuda").bfloat16() for n in (Nq, Nk, Nk))
    o, lse, _, ws = av.avsa_cross_attn_scores(q, k, v)
    o2, lse2, _, ws2 = av.avsa_cross_attn_scores(q, k, v, want_scores=False)
    for x in (ws, ws2):
        _status_ok(x)
    assert torch.equal(o, o2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("reverse", [False, True])
def test_cross_attention_row_maxima_growing_along_the_key_axis(reverse):
    """Pass 1 runs on the fast kernel too (key axis split across work items, or one item per query tile in the
    reverse direction): with logits that grow steeply from key block to key block its rows outgrow their
    first-tile reference and the exact-rescaling kernel must take the items over."""
    import dataclasses
    w = dataclasses.replace(wl.WORKLOADS["medium128"], H=12)      # forward: 24 query tiles -> key splits of 3 tiles
    qa, kc, vc = wl.make_cross_qkv(w, 3)
    if reverse:
        qa, kc, vc = kc, torch.cat([qa] * 5, dim=2), torch.cat([qa] * 5, dim=2).flip(2)   # 2070 queries, 360 keys
    u = 1.0 / np.sqrt(w.d)
    qa = (qa.float() + 8.0 * u).to(torch.bfloat16)
    nk = kc.shape[2]
    ramp = torch.arange(nk, dtype=torch.float32).div(w.blk, rounding_mode="floor") * (80.0 if reverse else 48.0)
    kc = (kc.float() + (ramp * u).view(1, 1, -1, 1)).to(torch.bfloat16)
    o, lse, _, ws = av.avsa_cross_attn_scores(qa.cuda(), kc.cuda(), vc.cuda(), want_scores=False)
    _status_ok(ws)
    assert av.avsa_redo_count(ws) > 0
    want_o, want_lse, _ = orc.cross_attention(_np64(qa), _np64(kc), _np64(vc))
    _close(_np64(o), want_o, "growing maxima cross O")
    _close_lse(_np64(lse), want_lse, "growing maxima cross lse")


def test_cross_attention_scores_need_one_short_axis():
    """Neither the queries nor the keys of a head fit on chip: the score pass is refused on the host."""
    q = torch.zeros((1, 1, 1024, 128), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(av.AvsaError) as e:
        av.avsa_cross_attn_scores(q, q, q)
    assert e.value.status == av.AVSA_ERR_UNSUPPORTED
    o, lse, s, ws = av.avsa_cross_attn_scores(q, q, q, want_scores=False)  # outputs alone are fine
    _status_ok(ws)


# ------------------------------------------------------------------------------------------- whole path
def test_whole_path_tiny_matches_oracle():
    w = wl.WORKLOADS["tiny"]
    qa, kc, vc = (t.cuda() for t in wl.make_cross_qkv(w, 0))
    q, k, v = (t.cuda() for t in wl.make_self_qkv(w, 0))
    n_protect = av.avsa_count_from_percent(w.protect_pct, w.n_video)
    k_keep = av.avsa_count_from_percent(w.keep_pct, w.n_blocks)
    assert (n_protect, k_keep) == (26, 2)
    _, _, s, _ = av.avsa_cross_attn_scores(qa, kc, vc, score_gamma=1.0 / (w.H * w.n_audio))
    m = av.avsa_build_block_mask(q, k, s, n_protect, k_keep, w.blk)
    o, _, ws = av.avsa_sparse_self_attn(q, k, v, m["col_idx"], m["col_cnt"], w.blk)
    _status_ok(ws)
    assert av.avsa_redo_count(ws) == 0            # unit-variance logits never outgrow the first-tile reference
    # oracle end to end
    _, _, A = orc.cross_attention(_np64(qa), _np64(kc), _np64(vc))
    s64 = orc.column_scores(A, gamma=1.0 / (w.H * w.n_audio))
    bs64 = orc.block_scores(_np64(q), _np64(k), w.blk)
    idx, cnt, ptok, pblk = orc.build_block_mask(bs64, s64, n_protect, k_keep, w.blk, w.n_video)
    region = wl.region_mask(w, "cpu").numpy()
    assert (ptok[0].astype(bool) & region).sum() >= 24                    # the planted region is what gets protected
    # the planted margin makes the selections agree exactly between fp32/bf16 GPU scores and fp64 oracle
    assert np.array_equal(m["prot_blk"].cpu().numpy(), pblk)
    assert np.array_equal(m["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(m["col_idx"].cpu().numpy(), idx)
    want, _ = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, w.blk)
    _close(_np64(o), want, "whole path O")


@pytest.mark.parametrize("name", ["tiny", "medium128"])
def test_whole_path_replays_from_a_cuda_graph(name):
    """The calls only enqueue work on the given stream (no allocation, no synchronisation, no host read of
    device data), so one layer-step can be captured into a CUDA graph once and replayed on new inputs.
    The replays must reproduce the eager results bit for bit, and the eager results are held to the oracle."""
    w = wl.WORKLOADS[name]
    n_protect = av.avsa_count_from_percent(w.protect_pct, w.n_video)
    k_keep = av.avsa_count_from_percent(w.keep_pct, w.n_blocks)
    gamma = 1.0 / (w.H * w.n_audio)

    def inputs(seed):
        return [t.cuda() for t in wl.make_cross_qkv(w, seed)] + [t.cuda() for t in wl.make_self_qkv(w, seed)]

    def eager(qa, kc, vc, q, k, v):
        _, _, s, _ = av.avsa_cross_attn_scores(qa, kc, vc, score_gamma=gamma, want_o=False)
        m = av.avsa_build_block_mask(q, k, s, n_protect, k_keep, w.blk)
        o, lse, ws = av.avsa_sparse_self_attn(q, k, v, m["col_idx"], m["col_cnt"], w.blk, want_lse=True)
        _status_ok(ws)
        return s, m, o, lse

    static = [t.clone() for t in inputs(0)]
    qa, kc, vc, q, k, v = static
    s0, m0, o0, lse0 = eager(*static)                       # also the warm-up that loads every kernel
    # caller-owned buffers of the captured step
    s = torch.empty_like(s0)
    lse_a = torch.empty((w.B, w.H, w.n_audio), dtype=torch.float32, device="cuda")
    out = {key: torch.empty_like(m0[key]) for key in ("block_scores", "col_idx", "col_cnt", "prot_tok", "prot_blk")}
    o, lse = torch.empty_like(o0), torch.empty_like(lse0)
    ws_c = torch.empty(av.avsa_cross_attn_scores_workspace_bytes(w.B, w.H, w.n_audio, w.n_video, w.d), dtype=torch.uint8, device="cuda")
    ws_m = torch.empty(av.avsa_build_block_mask_workspace_bytes(w.B, w.H, w.n_video, w.d, w.blk), dtype=torch.uint8, device="cuda")
    ws_a = torch.empty(av.avsa_sparse_self_attn_workspace_bytes(w.B, w.H, w.n_video, w.d, w.blk), dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        av.avsa_cross_attn_scores(qa, kc, vc, scores=s, score_gamma=gamma, want_o=False, lse=lse_a, ws=ws_c)
        av.avsa_build_block_mask(q, k, s, n_protect, k_keep, w.blk, out=out, ws=ws_m)
        av.avsa_sparse_self_attn(q, k, v, out["col_idx"], out["col_cnt"], w.blk, o=o, lse=lse, ws=ws_a)
    for seed in (0, 5, 0):
        fresh = inputs(seed)
        for dst, src in zip(static, fresh):
            dst.copy_(src)
        for t in (s, o, lse, out["col_idx"], out["col_cnt"]):
            t.fill_(0)
        graph.replay()
        torch.cuda.synchronize()
        for ws_x in (ws_c, ws_m, ws_a):
            _status_ok(ws_x)
        assert av.avsa_redo_count(ws_a) == 0
        want_s, want_m, want_o, want_lse = eager(*fresh)
        assert torch.equal(s, want_s), f"seed {seed}: scores differ between replay and eager call"
        for key in ("col_idx", "col_cnt", "prot_tok", "prot_blk", "block_scores"):
            assert torch.equal(out[key], want_m[key]), f"seed {seed}: {key} differs between replay and eager call"
        assert torch.equal(o.view(torch.int16), want_o.view(torch.int16)), f"seed {seed}: O differs"
        assert torch.equal(lse, want_lse), f"seed {seed}: LSE differs"
    # the eager results of the last seed against the oracle
    idx, cnt = out["col_idx"].cpu().numpy(), out["col_cnt"].cpu().numpy()
    want, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, w.blk)
    _close(_np64(o), want, "graph replay O")
    _close_lse(_np64(lse), want_l, "graph replay lse")


# ------------------------------------------------------------------------------------------- token-exact protection
@pytest.mark.parametrize("name", ["tiny", "small128", "medium128"])
def test_token_exact_protection_matches_oracle(name):
    w = wl.WORKLOADS[name]
    q, k, v = wl.make_self_qkv(w, 6)
    _, _, _, s64 = _oracle_scores(w, 6)
    n_protect = orc.ceil_pct(w.protect_pct, w.n_video)
    k_keep = max(1, orc.ceil_pct(w.keep_pct, w.n_blocks))
    bs32 = orc.block_scores(_np64(q), _np64(k), w.blk).astype(np.float32)
    s32 = s64.astype(np.float32)
    idx, cnt, ptok, _ = orc.build_block_mask(bs32, s32, n_protect, k_keep, w.blk, w.n_video, protect_rows=False)
    m = av.avsa_build_block_mask(None, None, torch.from_numpy(s32).cuda(), n_protect, k_keep, w.blk,
                                 flags=av.AVSA_PROTECT_TOKENS | av.AVSA_USE_GIVEN_BLOCK_SCORES,
                                 block_scores=torch.from_numpy(bs32).cuda(), shape=(w.B, w.H, w.n_video, w.d))
    assert np.array_equal(m["col_idx"].cpu().numpy(), idx) and np.array_equal(m["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(m["prot_tok"].cpu().numpy(), ptok)
    assert (cnt == k_keep).all()                                       # no block is made dense
    qc, kc, vc = q.cuda(), k.cuda(), v.cuda()
    o, lse, ws = av.avsa_sparse_self_attn(qc, kc, vc, m["col_idx"], m["col_cnt"], w.blk, want_lse=True)
    _status_ok(ws)
    ws2 = av.avsa_protected_rows_attn(qc, kc, vc, m["prot_tok"], n_protect, w.blk, o, lse=lse)
    _status_ok(ws2)
    want_o, want_l = orc.protected_attention_token_exact(_np64(q), _np64(k), _np64(v), idx, cnt, ptok, w.blk)
    _close(_np64(o), want_o, f"{name} token-exact O")
    _close_lse(_np64(lse), want_l, f"{name} token-exact lse")
    # a flag count that disagrees with n_protect is refused on the device and nothing is overwritten
    before = o.clone()
    ws3 = av.avsa_protected_rows_attn(qc, kc, vc, m["prot_tok"], n_protect + 1, w.blk, o)
    code, detail = av.avsa_read_status(ws3)
    assert code == av.AVSA_ERR_BAD_MASK and detail[2] == n_protect
    assert torch.equal(before, o)
    # zero protected tokens: a no-op
    av.avsa_protected_rows_attn(qc, kc, vc, torch.zeros_like(m["prot_tok"]), 0, w.blk, o)
    torch.cuda.synchronize()
    assert torch.equal(before, o)


# ------------------------------------------------------------------------------------------- Eq. 12-15
@pytest.mark.parametrize("Nv,Na,C", [(390, 40, 384), (2070, 72, 512), (5, 3, 8)])
def test_cache_indicators_match_oracle(Nv, Na, C):
    B = 2
    g = torch.Generator().manual_seed(Nv)
    y_v = torch.randn((B, Nv, C), generator=g).bfloat16()
    yhat_v = (y_v.float() + 0.2 * torch.randn((B, Nv, C), generator=g)).bfloat16()
    y_a = torch.randn((B, Na, C), generator=g).bfloat16()
    yhat_a = (y_a.float() + 0.05 * torch.randn((B, Na, C), generator=g)).bfloat16()
    prot = (torch.rand((B, Nv), generator=g) < 0.1).to(torch.uint8)
    prot[:, 0] = 1
    s_cur = torch.rand((B, Nv), generator=g)
    s_anchor = (s_cur + 0.3 * torch.rand((B, Nv), generator=g)).float()
    out, ws = av.avsa_cache_indicators(y_v.cuda(), yhat_v.cuda(), y_a.cuda(), yhat_a.cuda(), prot.cuda(), s_cur.cuda(),
                                       s_anchor.cuda())
    _status_ok(ws)
    got = out.cpu().numpy()
    for b in range(B):
        want = orc.cache_indicators(_np64(y_v[b]), _np64(yhat_v[b]), _np64(y_a[b]), _np64(yhat_a[b]), prot[b].numpy(),
                                    _np64(s_cur[b]), _np64(s_anchor[b]))
        for i, key in enumerate(("dv", "da", "dp", "ds", "dsync")):
            assert abs(got[b, i] - want[key]) <= 1e-4 * max(1.0, abs(want[key])), (b, key, got[b, i], want[key])
        assert bool(got[b, 5]) == want["reuse"]
    # no protected set and no saliency maps: those terms drop out
    out2, _ = av.avsa_cache_indicators(y_v.cuda(), y_v.cuda(), y_a.cuda(), y_a.cuda())
    assert np.allclose(out2.cpu().numpy()[:, :5], 0.0) and (out2.cpu().numpy()[:, 5] == 1.0).all()
    # reproducible bit for bit
    out3, _ = av.avsa_cache_indicators(y_v.cuda(), yhat_v.cuda(), y_a.cuda(), yhat_a.cuda(), prot.cuda(), s_cur.cuda(),
                                       s_anchor.cuda())
    assert torch.equal(out, out3)


@pytest.mark.parametrize("B,H,N,d,blk", [(1, 1, 1, 128, 128), (2, 1, 129, 128, 128), (3, 2, 65, 64, 64), (1, 5, 640, 128, 128)])
def test_degenerate_shapes_whole_path(B, H, N, d, blk):
    """One token, a one-token tail block, several batch items, one head: every call against the oracle."""
    NB = (N + blk - 1) // blk
    _whole_path_case(B, H, N, d, blk, 7, min(N, 3), max(1, NB // 2), B * 1000 + N)


@pytest.mark.parametrize("seed", range(6))
def test_random_shapes_whole_path(seed):
    """Seeded random batch, heads, lengths (video and audio), tile size, protected count and kept count: every
    call of the path against the oracle, block-level and token-exact protection."""
    rng = np.random.default_rng(700 + seed)
    d = int(rng.choice([64, 128]))
    B, H = int(rng.integers(1, 3)), int(rng.integers(1, 5))
    N = int(rng.integers(2, 7 * d))
    NB = (N + d - 1) // d
    _whole_path_case(B, H, N, d, d, int(rng.integers(1, 300)), int(rng.integers(0, N // 4 + 2)),
                     int(rng.integers(1, NB + 1)), 800 + seed)


def _whole_path_case(B, H, N, d, blk, Na, n_protect, k_keep, seed):
    g = torch.Generator().manual_seed(seed)
    q, k, v = (torch.randn((B, H, N, d), generator=g).bfloat16() for _ in range(3))
    qa = torch.randn((B, H, Na, d), generator=g).bfloat16()
    gamma = 1.0 / (H * Na)
    o_a, lse_a, s, ws = av.avsa_cross_attn_scores(qa.cuda(), k.cuda(), v.cuda(), score_gamma=gamma)
    _status_ok(ws)
    want_oa, want_la, A = orc.cross_attention(_np64(qa), _np64(k), _np64(v))
    _close(_np64(o_a), want_oa, "cross O")
    _close_lse(_np64(lse_a), want_la, "cross lse")
    want_s = orc.column_scores(A, gamma=gamma)
    _close_scores(_np64(s), want_s, "scores")
    m = av.avsa_build_block_mask(q.cuda(), k.cuda(), s, n_protect, k_keep, blk)
    idx, cnt, ptok, pblk = orc.build_block_mask(m["block_scores"].cpu().numpy(), s.cpu().numpy(), n_protect, k_keep, blk, N)
    want_bs = orc.block_scores(_np64(q), _np64(k), blk)
    assert np.abs(m["block_scores"].cpu().numpy() - want_bs).max() <= 1e-4 * max(1.0, np.abs(want_bs).max())
    assert np.array_equal(m["col_idx"].cpu().numpy(), idx) and np.array_equal(m["col_cnt"].cpu().numpy(), cnt)
    assert np.array_equal(m["prot_tok"].cpu().numpy(), ptok) and np.array_equal(m["prot_blk"].cpu().numpy(), pblk)
    o, lse, ws3 = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), m["col_idx"], m["col_cnt"], blk, want_lse=True)
    _status_ok(ws3)
    want_o, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, blk)
    _close(_np64(o), want_o, "O")
    _close_lse(_np64(lse), want_l, "lse")
    # token-exact variant on the same inputs
    m2 = av.avsa_build_block_mask(q.cuda(), k.cuda(), s, n_protect, k_keep, blk, flags=av.AVSA_PROTECT_TOKENS)
    o2, lse2, _ = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), m2["col_idx"], m2["col_cnt"], blk, want_lse=True)
    ws4 = av.avsa_protected_rows_attn(q.cuda(), k.cuda(), v.cuda(), m2["prot_tok"], n_protect, blk, o2, lse=lse2)
    _status_ok(ws4)
    idx2, cnt2, ptok2, _ = orc.build_block_mask(m2["block_scores"].cpu().numpy(), s.cpu().numpy(), n_protect, k_keep, blk, N,
                                                protect_rows=False)
    want_o2, want_l2 = orc.protected_attention_token_exact(_np64(q), _np64(k), _np64(v), idx2, cnt2, ptok2, blk)
    _close(_np64(o2), want_o2, "token-exact O")
    _close_lse(_np64(lse2), want_l2, "token-exact lse")


def test_audio_branch_short_sequences():
    """The audio branch (m = a in Eq. 8-10) is the same three calls on a short sequence: fewer tokens than one
    block, and a two-block sequence with one protected block."""
    for (H, d, blk, N, k_keep, n_protect) in ((2, 64, 64, 40, 1, 4), (3, 128, 128, 256, 1, 13)):
        g = torch.Generator().manual_seed(N)
        q, k, v = (torch.randn((1, H, N, d), generator=g).bfloat16() for _ in range(3))
        s = torch.rand((1, N), generator=g)
        m = av.avsa_build_block_mask(q.cuda(), k.cuda(), s.cuda(), n_protect, k_keep, blk)
        idx, cnt, ptok, pblk = orc.build_block_mask(m["block_scores"].cpu().numpy(), s.numpy(), n_protect, k_keep, blk, N)
        assert np.array_equal(m["col_idx"].cpu().numpy(), idx) and np.array_equal(m["col_cnt"].cpu().numpy(), cnt)
        assert np.array_equal(m["prot_tok"].cpu().numpy(), ptok) and ptok.sum() == n_protect
        o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), m["col_idx"], m["col_cnt"], blk, want_lse=True)
        _status_ok(ws)
        want_o, want_l = orc.masked_attention(_np64(q), _np64(k), _np64(v), idx, cnt, blk)
        _close(_np64(o), want_o, f"audio branch N={N} O")
        _close_lse(_np64(lse), want_l, f"audio branch N={N} lse")


def test_host_side_argument_errors():
    w = wl.WORKLOADS["tiny"]
    q, k, v = (t.cuda() for t in wl.make_self_qkv(w, 0))
    NB = w.n_blocks
    idx = torch.zeros((1, 2, NB, NB), dtype=torch.int32, device="cuda")
    cnt = torch.ones((1, 2, NB), dtype=torch.int32, device="cuda")
    with pytest.raises(av.AvsaError) as e:
        av.avsa_sparse_self_attn(q, k, v, idx, cnt, 32)
    assert e.value.status == av.AVSA_ERR_UNSUPPORTED
    with pytest.raises(av.AvsaError) as e:
        av.avsa_sparse_self_attn(q, k, v, idx, cnt, w.blk, ws=torch.empty(256, dtype=torch.uint8, device="cuda")[:8])
    assert e.value.status == av.AVSA_ERR_WORKSPACE
    with pytest.raises(av.AvsaError) as e:
        av.avsa_build_block_mask(q, k, None, 3, 1, w.blk)
    assert e.value.status == av.AVSA_ERR_INVALID_ARG
    with pytest.raises(av.AvsaError) as e:
        av.avsa_build_block_mask(q, k, None, 0, NB + 1, w.blk)
    assert e.value.status == av.AVSA_ERR_INVALID_ARG


# ------------------------------------------------------------------------------------------- caller-owned scratch
def test_workspace_sizes_are_the_same_wherever_they_are_asked():
    """How short cross-attention runs depends on what the device can hold; its workspace does not: the sizes are those of a process
    that sees no device, every call of the shape is content with them, and asking makes no context on the device."""
    shapes = [(1, 8, 72, 2048, 128), (1, 24, 109, 1100, 128), (2, 3, 140, 333, 64), (1, 48, 100, 400, 128), (1, 74, 128, 512, 128), (1, 7, 128, 4096, 128),
              (1, 9, 128, 4096, 128), (1, 2, 72, 300, 128), (1, 24, 256, 32760, 128)]
    code = f"""if True:
        import ctypes
        from paper_2608_15522_b200 import binding as av
        print([av.avsa_cross_attn_scores_workspace_bytes(*s) for s in {shapes}])
        cu, flags, active = ctypes.CDLL("libcuda.so.1"), ctypes.c_uint(), ctypes.c_int()
        assert cu.cuInit(0) != 0 or cu.cuDevicePrimaryCtxGetState(0, ctypes.byref(flags), ctypes.byref(active)) == 0
        assert active.value == 0, "a context was made"
    """
    seen = []
    for env in ({}, {"CUDA_VISIBLE_DEVICES": ""}):
        r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env={**os.environ, **env}, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        assert r.returncode == 0, r.stdout
        seen.append(r.stdout.strip())
    assert seen[0] == seen[1] == str([av.avsa_cross_attn_scores_workspace_bytes(*s) for s in shapes])
    for (B, H, Nq, Nk, d), n in zip(shapes, eval(seen[0])):
        q, k = (torch.zeros((B, H, x, d), dtype=torch.bfloat16, device="cuda") for x in (Nq, Nk))
        for scores in (True, False):
            _status_ok(av.avsa_cross_attn_scores(q, k, k, want_scores=scores, ws=torch.empty(n, dtype=torch.uint8, device="cuda"))[3])


@pytest.mark.parametrize("offset", [4, 16])
def test_workspaces_cut_out_of_an_arena(offset):
    """Workspaces at 4 and 16 bytes from an aligned address: the bits of the aligned call, or refused where wider accesses are made.  Short
    cross-attention against more than 256 keys goes another way there (the sliced one writes parts of O 32 bytes at a time): the
    same within the bars, or refused where that way cuts rows too."""
    g = torch.Generator(device="cuda").manual_seed(4)
    R = lambda *s: torch.randn(s, generator=g, device="cuda").bfloat16()

    def check(call, nbytes, takes, exact=True):
        """`takes`: the alignment that the call takes (None: either way)."""
        n = max(nbytes, 256)
        ws = torch.empty(n + 32, dtype=torch.uint8, device="cuda")[offset:offset + n]
        assert ws.data_ptr() % 32 == offset
        try:
            got = call(ws)
        except av.AvsaError as e:
            assert e.status == av.AVSA_ERR_INVALID_ARG and (takes is None or offset % takes != 0)
            return
        assert takes is None or offset % takes == 0
        _status_ok(ws)
        for x, y in zip(call(None), got):
            assert torch.equal(x, y) if exact else (x.float() - y.float()).abs().max() <= 2e-2      # (O; LSE and scores differ less)

    for H, N, d in ((3, 700, 128), (5, 64 * 70 + 9, 64), (2, 300, 64)):
        q, k, v = R(1, H, N, d), R(1, H, N, d), R(1, H, N, d)
        s = torch.rand((1, N), generator=g, device="cuda")
        NB, n_protect = (N + d - 1) // d, N // 9
        names = ("block_scores", "col_idx", "col_cnt", "prot_tok", "prot_blk")
        mask = lambda ws, **kw: [av.avsa_build_block_mask(q, k, s, n_protect, max(1, NB // 4), d, ws=ws, **kw)[x] for x in names]
        m, n = mask(None), av.avsa_build_block_mask_workspace_bytes(1, H, N, d, d)
        check(mask, n, 4 if N == 300 else 16)
        check(lambda ws: mask(ws, block_scores=m[0], flags=av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES), n, 4)
        check(lambda ws: av.avsa_sparse_self_attn(q, k, v, m[1], m[2], d, want_lse=True, ws=ws)[:2],
              av.avsa_sparse_self_attn_workspace_bytes(1, H, N, d, d), 4)

        def rows(ws):
            o = torch.zeros_like(q)
            av.avsa_protected_rows_attn(q, k, v, m[3], n_protect, d, o, ws=ws)
            return (o,)
        check(rows, av.avsa_protected_rows_attn_workspace_bytes(1, H, N, d, d, n_protect), 16 if offset < 16 else None)
    for B, H, Nq, Nk, d, takes in ((1, 3, 700, 200, 128, 4), (2, 3, 140, 333, 64, None), (1, 40, 100, 400, 128, None), (1, 2, 60, 9000, 64, 32)):
        q, k, v = R(B, H, Nq, d), R(B, H, Nk, d), R(B, H, Nk, d)
        check(lambda ws: av.avsa_cross_attn_scores(q, k, v, ws=ws, score_gamma=1.0 / (H * Nq))[:3],
              av.avsa_cross_attn_scores_workspace_bytes(B, H, Nq, Nk, d), takes, exact=Nk <= 256)
    y = [R(1, 64, 64) for _ in range(4)]
    check(lambda ws: av.avsa_cache_indicators(*y, ws=ws)[:1], av.avsa_cache_indicators_workspace_bytes(1, 64, 64, 64), 16)


@pytest.mark.parametrize("name", ["tiny", "medium128"])
def test_results_do_not_depend_on_what_the_buffers_held_before(name):
    """Workspaces and outputs are caller-owned and arrive with arbitrary contents: every call must produce the
    same bits whether they were zero-filled or filled with 0xFF bytes (NaN patterns, negative counts)."""
    w = wl.WORKLOADS[name]
    qa, kc, vc = (t.cuda() for t in wl.make_cross_qkv(w, 3))
    q, k, v = (t.cuda() for t in wl.make_self_qkv(w, 3))
    n_protect = av.avsa_count_from_percent(w.protect_pct, w.n_video)
    k_keep = av.avsa_count_from_percent(w.keep_pct, w.n_blocks)
    NB = w.n_blocks
    C = w.H * w.d
    g = torch.Generator().manual_seed(9)
    y_v = torch.randn((w.B, w.n_video, C), generator=g).bfloat16().cuda()
    yhat_v = (y_v.float() * 1.1).bfloat16()
    y_a = torch.randn((w.B, w.n_audio, C), generator=g).bfloat16().cuda()
    yhat_a = (y_a.float() * 0.9).bfloat16()

    def run(fill):
        def buf(shape, dtype):
            t = torch.empty(shape, dtype=dtype, device="cuda")
            t.view(torch.uint8).fill_(fill)
            return t

        def scratch(nbytes):
            return buf((max(int(nbytes), 256),), torch.uint8)

        res = {}
        o_a, lse_a, s = buf(qa.shape, torch.bfloat16), buf(qa.shape[:3], torch.float32), buf((w.B, w.n_video), torch.float32)
        ws = scratch(av.avsa_cross_attn_scores_workspace_bytes(w.B, w.H, w.n_audio, w.n_video, w.d))
        av.avsa_cross_attn_scores(qa, kc, vc, scores=s, score_beta=0.0, score_gamma=1.0 / (w.H * w.n_audio), o=o_a,
                                  lse=lse_a, ws=ws)
        _status_ok(ws)
        res.update(o_a=o_a, lse_a=lse_a, s=s)
        for tag, flags in (("rows", av.AVSA_PROTECT_ROWS), ("tok", av.AVSA_PROTECT_TOKENS),
                           ("sum", av.AVSA_PROTECT_ROWS | av.AVSA_PROTECT_BLOCK_SUM)):
            out = dict(block_scores=buf((w.B, w.H, NB, NB), torch.float32), col_idx=buf((w.B, w.H, NB, NB), torch.int32),
                       col_cnt=buf((w.B, w.H, NB), torch.int32), prot_tok=buf((w.B, w.n_video), torch.uint8),
                       prot_blk=buf((w.B, NB), torch.uint8))
            ws = scratch(av.avsa_build_block_mask_workspace_bytes(w.B, w.H, w.n_video, w.d, w.blk))
            n = n_protect if tag != "sum" else max(1, NB // 4)
            av.avsa_build_block_mask(q, k, s, n, k_keep, w.blk, flags=flags, out=out, ws=ws)
            _status_ok(ws)
            for key, val in out.items():
                res[f"{tag}.{key}"] = val
        o, lse = buf(q.shape, torch.bfloat16), buf(q.shape[:3], torch.float32)
        ws = scratch(av.avsa_sparse_self_attn_workspace_bytes(w.B, w.H, w.n_video, w.d, w.blk))
        av.avsa_sparse_self_attn(q, k, v, res["tok.col_idx"], res["tok.col_cnt"], w.blk, o=o, lse=lse, ws=ws)
        _status_ok(ws)
        res.update(o_base=o.clone(), lse_base=lse.clone())
        ws = scratch(av.avsa_protected_rows_attn_workspace_bytes(w.B, w.H, w.n_video, w.d, w.blk, n_protect))
        av.avsa_protected_rows_attn(q, k, v, res["tok.prot_tok"], n_protect, w.blk, o, lse=lse, ws=ws)
        _status_ok(ws)
        res.update(o=o, lse=lse)
        ind = buf((w.B, 8), torch.float32)
        ws = scratch(av.avsa_cache_indicators_workspace_bytes(w.B, w.n_video, w.n_audio, C))
        av.avsa_cache_indicators(y_v, yhat_v, y_a, yhat_a, res["tok.prot_tok"], s, s, out=ind, ws=ws)
        _status_ok(ws)
        res["indicators"] = ind[:, :6].clone()
        torch.cuda.synchronize()
        return res

    a, b = run(0x00), run(0xFF)
    for key in a:
        assert torch.equal(a[key].view(torch.uint8), b[key].view(torch.uint8)), f"{key} depends on earlier buffer contents"


# ------------------------------------------------------------------------------------------- time-limited waits
def test_a_wait_that_nothing_ends_times_out_and_leaves_the_context_usable():
    """Every wait inside the tile kernels is time-limited.  The self-test kernel waits on a barrier that nothing
    signals: it must give up after the limit, report AVSA_ERR_TIMEOUT through the status record, and the next
    ordinary call on the same context must work."""
    ws = torch.empty(av.AVSA_STATUS_BYTES, dtype=torch.uint8, device="cuda")
    limit = 2_000_000                                           # about a millisecond
    av.avsa_selftest_bounded_wait(ws, limit)
    code, (where, item, waited_k) = av.avsa_read_status(ws)
    assert code == av.AVSA_ERR_TIMEOUT and where == 99 and item == 0
    assert limit // 1024 <= waited_k <= 4 * limit // 1024
    assert "timed out" in av.status_string(code)
    with pytest.raises(av.AvsaError):
        av.avsa_selftest_bounded_wait(ws, 3_000_000_000)        # limits beyond about a second are refused
    w = wl.WORKLOADS["tiny"]
    NB = w.n_blocks
    idx = np.broadcast_to(np.arange(NB, dtype=np.int32), (w.B, w.H, NB, NB)).copy()
    _run_sparse_case(w, 1, idx, np.full((w.B, w.H, NB), NB, np.int32))


@pytest.mark.parametrize("B,H,N,d,n_protect", [(2, 1, 1007, 64, 37), (2, 2, 513, 128, 1), (1, 3, 2600, 64, 700), (3, 1, 130, 128, 130)])
def test_protected_rows_odd_lengths(B, H, N, d, n_protect):
    """Flags at any alignment (odd N, several batch items), one to all rows: the flagged rows are dense rows, the others
    stay as they were, with and without an LSE."""
    g = torch.Generator().manual_seed(N + n_protect)
    q, k, v = (torch.randn((B, H, N, d), generator=g).to(torch.bfloat16) for _ in range(3))
    flags = torch.zeros((B, N), dtype=torch.uint8)
    for b in range(B):
        flags[b, torch.randperm(N, generator=g)[:n_protect]] = 1
    o = torch.full((B, H, N, d), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H, N), 7.0, dtype=torch.float32, device="cuda")
    ws = av.avsa_protected_rows_attn(q.cuda(), k.cuda(), v.cuda(), flags.cuda(), n_protect, d, o, lse=lse)
    _status_ok(ws)
    want_o, want_l = orc.dense_attention(_np64(q), _np64(k), _np64(v))
    on = flags.bool().numpy()[:, None, :].repeat(H, axis=1)
    got_o, got_l = _np64(o), _np64(lse)
    _close(got_o[on], want_o[on], "protected rows O")
    _close_lse(got_l[on], want_l[on], "protected rows lse")
    assert (got_o[~on] == 7.0).all() and (got_l[~on] == 7.0).all()


@pytest.mark.parametrize("heads,d,repeat", [(20, 128, 1), (40, 128, 5), (8, 64, 1), (20, 64, 5)])
def test_rows_that_outgrow_their_reference_in_short_and_long_calls(heads, d, repeat):
    """Steeply growing logits: a short call recomputes such items inside the tile kernel, a long one in a grid of its
    own (more than 64 tile pairs per SM, 32 without lists); list and range modes, both tile shapes of either."""
    n, na = 2070, 300
    g = torch.Generator().manual_seed(heads)
    q, k, v = (torch.randn((1, heads, n, d), generator=g) for _ in range(3))
    u = 1.0 / np.sqrt(d)
    q = (q + 8.0 * u).to(torch.bfloat16)
    ramp = torch.arange(n, dtype=torch.float32).div(d, rounding_mode="floor") * 16.0
    k = (k + (ramp * u).view(1, 1, -1, 1)).to(torch.bfloat16)
    v = v.to(torch.bfloat16)
    NB = (n + d - 1) // d
    idx = np.broadcast_to(np.arange(NB, dtype=np.int32), (1, heads, NB, NB)).copy()
    cnt = np.full((1, heads, NB), NB, np.int32)
    cnt[:, :, ::2] = 3
    o, lse, ws = av.avsa_sparse_self_attn(q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(idx).cuda(),
                                          torch.from_numpy(cnt).cuda(), d, want_lse=True)
    _status_ok(ws)
    n_redo, items = av.avsa_sparse_self_attn_redo_items(ws)
    assert n_redo >= heads * (NB // 2) and len(set(items.tolist())) == n_redo
    hs = [0, heads - 1]
    want_o, want_l = orc.masked_attention(_np64(q)[:, hs], _np64(k)[:, hs], _np64(v)[:, hs], idx[:, hs], cnt[:, hs], d)
    _close(_np64(o)[:, hs], want_o, "outgrown O")
    _close_lse(_np64(lse)[:, hs], want_l, "outgrown lse")
    qa = q[:, :, :na].contiguous()
    kc, vc = (torch.cat([t] * repeat, dim=2) for t in (k, v))
    oc, lc, _, wc = av.avsa_cross_attn_scores(qa.cuda(), kc.cuda(), vc.cuda(), want_scores=False)
    _status_ok(wc)
    assert av.avsa_redo_count(wc) > 0
    want_o, want_l, _ = orc.cross_attention(_np64(qa)[:, hs], _np64(kc)[:, hs], _np64(vc)[:, hs])
    _close(_np64(oc)[:, hs], want_o, "outgrown cross O")
    _close_lse(_np64(lc)[:, hs], want_l, "outgrown cross lse")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H,N,n_protect,short", [
    (8, 2600, 700, True),       # query tiles in parts of 7 key tiles, recomputed inside the tile kernel
    (40, 2070, 300, True),      # whole rows stored through the row map, inside the tile kernel
    (128, 768, 700, True),      # the same with the query tiles off the queue
    (64, 1500, 1500, False),    # whole rows, in the grid behind it
    (54, 2688, 2500, False),    # the queue with its end cut: whole rows and parts, in the grid behind it
])
def test_protected_rows_that_outgrow_their_reference(H, N, n_protect, short, d):
    """Dense rows whose logits grow by some 16 per 128 keys, in every form that their exact recomputation takes: the flagged
    rows are the oracle's, the others stay as they were."""
    assert (2 * H * -(-n_protect // 128) * -(-N // 128) <= 64 * 148) == short
    g = torch.Generator(device="cuda").manual_seed(N + d)
    q, k, v = (torch.randn((1, H, N, d), generator=g, device="cuda") for _ in range(3))
    u = 1.0 / np.sqrt(d)
    q = (q + 8.0 * u).to(torch.bfloat16)
    ramp = torch.arange(N, dtype=torch.float32, device="cuda").div(128, rounding_mode="floor") * 2.0 * np.sqrt(d)
    k = (k + (ramp * u).view(1, 1, -1, 1)).to(torch.bfloat16)
    v = v.to(torch.bfloat16)
    flags = torch.zeros((1, N), dtype=torch.uint8, device="cuda")
    flags[0, torch.randperm(N, generator=g, device="cuda")[:n_protect]] = 1
    o = torch.full((1, H, N, d), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((1, H, N), 7.0, dtype=torch.float32, device="cuda")
    ws = av.avsa_protected_rows_attn(q, k, v, flags, n_protect, d, o, lse=lse)
    _status_ok(ws)
    assert av.avsa_redo_count(ws) >= H * -(-n_protect // 128)      # every query tile, in one part at least
    hs, on = [0, H - 1], flags[0].bool().cpu().numpy()
    want_o, want_l = orc.dense_attention(_np64(q[:, hs]), _np64(k[:, hs]), _np64(v[:, hs]))
    got_o, got_l = _np64(o[:, hs]), _np64(lse[:, hs])
    _close(got_o[:, :, on], want_o[:, :, on], "outgrown protected O")
    _close_lse(got_l[:, :, on], want_l[:, :, on], "outgrown protected lse")
    off = ~flags[0].bool()
    assert bool((o[:, :, off] == 7.0).all()) and bool((lse[:, :, off] == 7.0).all())


@pytest.mark.parametrize("n", [1, 63, 256, 257, 511, 512, 513])
def test_mask_with_the_select_in_the_pooling_grid(n):
    """Up to 512 tokens one launch selects and pools: token flags and block flags are the oracle's, ties at the threshold included,
    block scores are its up to fp32 sums, and the lists hold the largest of the scores that the call returns."""
    B, H, d, n_protect = 3, 2, 64, max(1, n // 9)
    NB = (n + d - 1) // d
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k = (torch.randn((B, H, n, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    s = torch.round(torch.randn((B, n), generator=g, device="cuda") * 4) / 4
    k_keep = max(1, NB // 2)
    m = av.avsa_build_block_mask(q, k, s, n_protect, k_keep, d)
    _status_ok(m["ws"])
    want = orc.block_scores(_np64(q), _np64(k), d)
    _, _, tok, blk = orc.build_block_mask(want, s.cpu().numpy(), n_protect, k_keep, d, n)
    assert np.array_equal(m["prot_tok"].cpu().numpy(), tok) and np.array_equal(m["prot_blk"].cpu().numpy(), blk)
    bs, idx, cnt = (m[x].cpu().numpy() for x in ("block_scores", "col_idx", "col_cnt"))
    assert np.abs(bs - want).max() <= 1e-4 * np.abs(want).max()
    assert np.array_equal(cnt, np.broadcast_to(np.where(blk != 0, NB, k_keep)[:, None, :], cnt.shape))
    for row, scores_row, c in zip(idx.reshape(-1, NB), bs.reshape(-1, NB), cnt.reshape(-1)):
        kept = row[:c]
        assert (np.diff(kept) > 0).all() and (row[c:] == -1).all()
        rest = np.setdiff1d(np.arange(NB), kept)
        assert rest.size == 0 or scores_row[kept].min() >= scores_row[rest].max()


@pytest.mark.parametrize("d,n,heads", [(128, 1, 2), (128, 127, 3), (128, 129, 74), (128, 256, 5), (128, 257, 5), (128, 200, 75), (64, 65, 4),
                                       (64, 257, 3), (64, 320, 6), (64, 321, 6)])
@pytest.mark.parametrize("flags", [av.AVSA_PROTECT_ROWS, av.AVSA_PROTECT_ROWS | av.AVSA_PROTECT_COLS, av.AVSA_PROTECT_TOKENS])
def test_mask_of_a_short_sequence_in_one_launch(d, n, heads, flags):
    """A CTA per (batch, head) pair pools, selects, scores and lists: block counts that share the pooling warps unevenly, the last
    length of each head size and the next, as many heads as SMs and more, none protected, and [B,N,H,d] storage."""
    B, NB = 2, (n + d - 1) // d
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k = (torch.randn((B, n, heads, d), generator=g, device="cuda").bfloat16().transpose(1, 2) for _ in range(2))
    s = torch.round(torch.randn((B, n), generator=g, device="cuda") * 4) / 4
    k_keep = max(1, NB // 2)
    for n_protect in (0, max(1, n // 9)):
        m = av.avsa_build_block_mask(q, k, s if n_protect else None, n_protect, k_keep, d, flags=flags)
        _status_ok(m["ws"])
        want, got = orc.block_scores(_np64(q), _np64(k), d), m["block_scores"].cpu().numpy()
        assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max()      # (fp32 sums of 128 means and products)
        idx, cnt, tok, blk = orc.build_block_mask(got, s.cpu().numpy(), n_protect, k_keep, d, n,
                                                  protect_rows=bool(flags & av.AVSA_PROTECT_ROWS), protect_cols=bool(flags & av.AVSA_PROTECT_COLS))
        for key, x in (("col_idx", idx), ("col_cnt", cnt), ("prot_tok", tok), ("prot_blk", blk)):
            assert np.array_equal(m[key].cpu().numpy(), x), key


@pytest.mark.parametrize("NB", [1, 32, 33, 256, 257, 512, 513, 1024, 1025])
def test_mask_select_over_row_lengths(NB):
    """The select's key slots per lane at their limits: distinct scores, heavy ties, one bit of difference, a sign change,
    infinities and NaN, all with few and many kept."""
    blk = 64
    N = NB * blk - 3
    rng = np.random.default_rng(NB)
    bs = rng.standard_normal((1, 1, NB, NB)).astype(np.float32)
    for r, row in enumerate(bs[0, 0]):
        if r % 6 == 1:
            row[:] = rng.integers(0, 3, NB)
        elif r % 6 == 2:
            row[:] = 1.5
            row[rng.integers(NB)] = np.nextafter(np.float32(1.5), np.float32(2.0))
        elif r % 6 == 3:
            row[:] *= np.float32(1e-42)
        elif r % 6 == 4:
            row[rng.integers(NB)] = np.inf
            row[rng.integers(NB)] = -np.inf
            row[rng.integers(NB)] = np.nan
        elif r % 6 == 5:
            row[:] = -np.inf
    s = rng.random((1, N)).astype(np.float32)
    for k_keep in sorted({1, max(1, NB // 7), max(1, NB - 1), NB}):
        idx, cnt, _, _ = orc.build_block_mask(bs, s, 3, k_keep, blk, N)
        out = av.avsa_build_block_mask(None, None, torch.from_numpy(s).cuda(), 3, k_keep, blk,
                                       flags=av.AVSA_PROTECT_ROWS | av.AVSA_USE_GIVEN_BLOCK_SCORES,
                                       block_scores=torch.from_numpy(bs).cuda(), shape=(1, 1, N, 64))
        _status_ok(out["ws"])
        assert np.array_equal(out["col_cnt"].cpu().numpy(), cnt)
        assert np.array_equal(out["col_idx"].cpu().numpy(), idx)


@pytest.mark.parametrize("reverse", [False, True])
def test_host_threads_with_short_and_long_axes_do_not_disturb_each_other(reverse):
    """Two host threads, each with its stream, buffers and shape: both run the same score pass (272 and 512 queries the one with
    four reduction groups, 272 and 512 keys the reverse one), which needs more or less shared memory by the length of the axis
    that stays on chip (210 and 226 KB; 195 and 227 KB), and no call may fail because of what the other thread's last one asked
    for."""
    import threading
    shapes = ((272, 600), (512, 600))      # (short axis, long axis)
    inputs, want = [], []
    for n_short, n_long in shapes:
        g = torch.Generator(device="cuda").manual_seed(n_short)
        nq, nk = (n_long, n_short) if reverse else (n_short, n_long)
        q, k = (torch.randn((1, 1, n, 128), generator=g, device="cuda").bfloat16() for n in (nq, nk))
        buf = dict(scores=torch.empty((1, nk), device="cuda"), lse=torch.empty((1, 1, nq), device="cuda"),
                   ws=torch.empty(av.avsa_cross_attn_scores_workspace_bytes(1, 1, nq, nk, 128), dtype=torch.uint8, device="cuda"))
        inputs.append((q, k, buf))
        want.append(av.avsa_cross_attn_scores(q, k, k, want_o=False, **buf)[2].clone())
    torch.cuda.synchronize()
    failed = []

    def work(i):
        q, k, buf = inputs[i]
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for _ in range(2000):
                try:
                    av.avsa_cross_attn_scores(q, k, k, want_o=False, **buf)
                except av.AvsaError as e:
                    failed.append((i, str(e)))
                    break
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for (q, k, buf), w in zip(inputs, want):
        assert torch.equal(buf["scores"], w)


def test_a_refused_launch_fails_its_own_call_only():
    """65536 (batch, head) pairs are one more than the mask's pooling grid can have, which the launch itself reports.  The
    call fails; the thread's next call knows nothing of it (the indicators: their call sets no kernel attribute, which would
    clear the runtime's last error by itself)."""
    q = torch.zeros((1, 65536, 1, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(av.AvsaError) as e:
        av.avsa_build_block_mask(q, q, None, 0, 1, 64)
    assert e.value.status == av.AVSA_ERR_CUDA
    y = torch.ones((1, 8, 64), dtype=torch.bfloat16, device="cuda")
    out, ws = av.avsa_cache_indicators(y, y, y, y)
    _status_ok(ws)
    assert (out[0, :5] == 0.0).all() and out[0, 5] == 1.0


def test_a_refused_tensor_map_leaves_the_thread_its_context():
    """A head stride that no tensor map can hold is refused on the host with nothing enqueued; a thread that works in a context of its
    own still does so afterwards."""
    import ctypes
    import threading
    driver = ctypes.CDLL("libcuda.so.1")
    lib = av.load_library()
    t = torch.zeros((2, 64, 64), dtype=torch.bfloat16, device="cuda")
    lse, ws = torch.empty((2, 64), device="cuda"), torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    device = t.device.index
    seen = {}

    def work():
        own, current, dev = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_int()
        assert driver.cuDeviceGet(ctypes.byref(dev), device) == 0
        assert driver.cuCtxCreate_v2(ctypes.byref(own), 0, dev) == 0      # (and makes it current)
        far = av._Bf16Tensor4(t.data_ptr(), 0, 1 << 40, 64)
        seen["status"] = lib.avsa_cross_attn_scores(1, 2, 64, 64, 64, far, far, far, None, lse.data_ptr(), None, 0.0, 1.0, 0.0,
                                                    ws.data_ptr(), ws.numel(), None)
        assert driver.cuCtxGetCurrent(ctypes.byref(current)) == 0
        seen["kept"] = current.value == own.value
        assert driver.cuCtxDestroy_v2(own) == 0

    thread = threading.Thread(target=work)
    thread.start()
    thread.join()
    assert seen == {"status": av.AVSA_ERR_CUDA, "kept": True}


@pytest.mark.parametrize("growth", [0.0, 4.0])
def test_cross_attention_queue_with_its_end_cut(growth):
    """240 heads x 4 query tiles x 29 key tiles: long enough for the queue, whose last units are cut in two.  Whole query
    tiles go out as tiles, the cut ones through the merge, and the score pass takes the LSEs of both.  With logits that grow by
    4 per 128 keys whole items and parts (15 tiles) outgrow their reference and are recomputed."""
    B, H, nq, nk, d = 10, 24, 512, 3712, 64
    g = torch.Generator(device="cuda").manual_seed(17)
    u = 1.0 / np.sqrt(d)
    q, k, v = (torch.randn((B, H, n, d), generator=g, device="cuda") for n in (nq, nk, nk))
    if growth:
        q = q + 8.0 * u
        ramp = torch.arange(nk, dtype=torch.float32, device="cuda").div(128, rounding_mode="floor") * growth * np.sqrt(d) / 8.0
        k = k + (ramp * u).view(1, 1, -1, 1)
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    o, lse, s, ws = av.avsa_cross_attn_scores(q, k, v, score_gamma=1.0 / (H * nq))
    _status_ok(ws)
    assert (av.avsa_redo_count(ws) >= B * H * 4) if growth else (av.avsa_redo_count(ws) == 0)
    for b in (0, B - 1):      # whole rows; cut rows
        want_o, want_lse, A = orc.cross_attention(_np64(q[b : b + 1]), _np64(k[b : b + 1]), _np64(v[b : b + 1]))
        _close(_np64(o[b : b + 1]), want_o, "queue O")
        _close_lse(_np64(lse[b : b + 1]), want_lse, "queue lse")
        _close_scores(_np64(s[b : b + 1]), orc.column_scores(A, gamma=1.0 / (H * nq)), "queue scores")
    _, lse2, _, _ = av.avsa_cross_attn_scores(q, k, v, want_scores=False, want_o=False)
    assert torch.equal(lse, lse2)


@pytest.mark.parametrize("d", [64, 128])
def test_long_dense_rows_do_not_drift_towards_zero(d):
    """The tensor cores' fp32 accumulation truncates, so what one accumulator sums is bounded (64 key tiles, 32 with 64
    channels).  With values of mean 1 the error along the result shows it: 1.1e-4 to 1.3e-4 of the value in such runs, 2.4e-4
    when the 384 tiles of this sequence are one run; bf16 rounding averages out over the 32768 (16384) elements compared
    (1.8e-3 / sqrt(16384) = 1.4e-5)."""
    H, N, n_protect = 8, 49152, 8192
    g = torch.Generator(device="cuda").manual_seed(d)
    q, k, v = (torch.randn((1, H, N, d), generator=g, device="cuda") for _ in range(3))
    q, k, v = q.to(torch.bfloat16), k.to(torch.bfloat16), (v + 1.0).to(torch.bfloat16)
    rows = torch.randperm(N, generator=g, device="cuda")[:n_protect]
    flags = torch.zeros((1, N), dtype=torch.uint8, device="cuda")
    flags[0, rows] = 1
    o = torch.zeros_like(q)
    _status_ok(av.avsa_protected_rows_attn(q, k, v, flags, n_protect, d, o))
    hs, rows = [0, 1], rows[:128]      # (the last heads are the cut end of the queue)
    want, _, _ = orc.cross_attention(_np64(q[:, hs][:, :, rows]), _np64(k[:, hs]), _np64(v[:, hs]))
    got = _np64(o[:, hs][:, :, rows])
    _close(got, want, "long dense rows")
    drift = ((got - want) * want).sum() / (want * want).sum()
    assert abs(drift) <= 1.8e-4, f"drift {drift:.2e}"


# ------------------------------------------------------------------------------------------- whole calls in native code
@pytest.mark.parametrize("given", [False, True])
def test_whole_calls_give_what_the_general_way_gives(monkeypatch, given):
    """Plain tensors go through one native call a wrapper; the same calls the general way (as for any other class of tensor) give
    the same bits, objects that the caller brings come back as they are, and refusals are the same."""
    w = wl.WORKLOADS["tiny"]
    q, k, v = (t.cuda() for t in wl.make_self_qkv(w, 3))
    qa, kc, vc = (t.cuda() for t in wl.make_cross_qkv(w, 3))
    s = torch.rand((w.B, w.n_video), device="cuda")
    NB, N, n_protect = w.n_blocks, w.n_video, 20

    def layer():
        kw = [{}, {}, {}, {}]
        if given:
            kw = [dict(out=dict(block_scores=torch.empty((w.B, w.H, NB, NB), device="cuda"), prot_blk=torch.empty((w.B, NB), dtype=torch.uint8, device="cuda"))),
                  dict(o=torch.empty_like(q), lse=torch.empty((w.B, w.H, N), device="cuda")),
                  dict(scores=torch.full((w.B, N), 0.25, device="cuda"), score_beta=0.5, o=torch.empty_like(qa)),
                  dict(ws=torch.empty(av.avsa_protected_rows_attn_workspace_bytes(w.B, w.H, N, w.d, w.blk, n_protect), dtype=torch.uint8, device="cuda"))]
        m = av.avsa_build_block_mask(q, k, s, n_protect, 2, w.blk, flags=av.AVSA_PROTECT_TOKENS, **kw[0])
        o, lse, ws = av.avsa_sparse_self_attn(q, k, v, m["col_idx"], m["col_cnt"], w.blk, want_lse=True, **kw[1])
        wp = av.avsa_protected_rows_attn(q, k, v, m["prot_tok"], n_protect, w.blk, o, lse=lse, **kw[3])
        oc, lc, sc, wc = av.avsa_cross_attn_scores(qa, kc, vc, **kw[2])
        plain = av.avsa_cross_attn_scores(qa, kc, vc, want_o=False, want_scores=False)
        assert plain[0] is None and plain[2] is None
        if given:
            assert m["block_scores"] is kw[0]["out"]["block_scores"] and m["prot_blk"] is kw[0]["out"]["prot_blk"]
            assert o is kw[1]["o"] and lse is kw[1]["lse"] and oc is kw[2]["o"] and sc is kw[2]["scores"] and wp is kw[3]["ws"]
        for x in (m["ws"], ws, wp, wc, plain[3]):
            _status_ok(x)
        torch.cuda.synchronize()
        return [m[key].clone() for key in ("block_scores", "col_idx", "col_cnt", "prot_tok", "prot_blk")] + [o, lse, oc, lc, sc, plain[1]]

    def refusals():
        got = []
        for call in (lambda: av.avsa_sparse_self_attn(q, k, v, None, None, w.blk), lambda: av.avsa_sparse_self_attn(q.float(), k, v, q, q, w.blk),
                     lambda: av.avsa_build_block_mask(q[0], k, s, 1, 1, w.blk), lambda: av.avsa_build_block_mask(q, k, s, 1, 1, 64.5),
                     lambda: av.avsa_build_block_mask(q, k, s, N + 1, 1, w.blk), lambda: av.avsa_cross_attn_scores(qa, kc.cpu(), vc),
                     lambda: av.avsa_cross_attn_scores(qa, kc, vc, ws=torch.empty(256, dtype=torch.uint8, device="cuda"))):
            with pytest.raises(Exception) as e:
                call()
            got.append((e.type, str(e.value)))
        return got

    native, native_refusals = layer(), refusals()

    class General:
        empty, empty_as = av._alloc().empty, av._alloc().empty_as
        cross = mask = sparse = protected_rows = staticmethod(lambda *a: None)
    monkeypatch.setattr(av, "_alloc_module", General)
    for a, b in zip(native, layer()):
        assert a.dtype == b.dtype and a.shape == b.shape and a.stride() == b.stride() and torch.equal(a, b)
    assert native_refusals == refusals()
