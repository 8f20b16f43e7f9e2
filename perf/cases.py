"""Performance cases of the library: what a joint audio-video diffusion transformer asks of it, call by call.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the same ranges,
``prepare`` the tensors and buffers that a program holds before the call, ``run`` one pass through the public entry
points, ``work`` what that pass cannot do without, ``tolerance`` how far two correct implementations may be apart.

Kinds of pass
  layer       one dual-stream layer-step in the order of the method: block mask from the cached saliency, sparse video
              self-attention under it (and the dense rows of the protected tokens in token-exact mode), then the
              audio->video cross-attention that blends its response scores into the cache (Eq. 4)
  self        mask + sparse self-attention of one stream alone (the audio branch has no response scores of its own)
  cross       one direction of the bidirectional cross-attention, with or without the score pass
  mask        the block mask alone
  sparse      sparse self-attention alone, under given lists, with the log-sum-exp that a merge with another branch needs
  indicators  the cache-reuse indicators of Eq. 12-15
"""
from __future__ import annotations

import math
import random

import torch

from paper_2608_15522_b200 import binding as av
from paper_2608_15522_b200 import workloads as wl

# Every field a case may leave out.
DEFAULTS = {"B": 1, "H": 24, "d": 128, "frames": 1, "rows": 1, "cols": 1, "audio": 0, "keep_pct": 25, "protect_pct": 5,
            "protect": "blocks",      # blocks | tokens | cols (protected rows and columns) | sum (blocks by summed response)
            "layout": "bhnd",         # or bnhd: what a fused qkv projection leaves behind, read through strides
            "direction": "a2v",       # cross: audio queries over video keys, or v2a
            "update": True,           # cross: with the score pass (every K-th denoising step) or without
            "lse": False,             # sparse: with the log-sum-exp output
            "keep_buffers": True}     # the program keeps its outputs and workspaces (else the wrappers allocate them)


def _full(case):
    c = dict(DEFAULTS)
    c.update(case)
    return c


def _tokens(c):
    return c["frames"] * c["rows"] * c["cols"]


def listed():
    return [
        # The smallest layer-step: 256 video tokens, head size 64.  Launches and host time are all there is to it.
        {"name": "layer_tiny_d64", "kind": "layer", "H": 2, "d": 64, "frames": 4, "rows": 8, "cols": 8, "audio": 32,
         "keep_pct": 50, "protect_pct": 10},
        # A preview-size clip in a batch of two (conditional and unconditional branch), ragged last block (2070 tokens).
        {"name": "layer_preview_batch2", "kind": "layer", "B": 2, "H": 4, "frames": 5, "rows": 18, "cols": 23, "audio": 72},
        # The audio stream's own self-attention: one to four blocks per head, called straight, nothing preallocated.
        {"name": "self_audio_branch", "kind": "self", "cols": 157, "keep_pct": 50, "keep_buffers": False},
        # Mid-length layer-step (17856 tokens), token-exact protection.
        {"name": "layer_mid_tokens", "kind": "layer", "frames": 31, "rows": 24, "cols": 24, "audio": 160, "protect": "tokens"},
        # The usual 5-second layer-step (32760 tokens), block protection: the benchmark's default workload.
        {"name": "layer_ovi_blocks", "kind": "layer", "frames": 21, "rows": 30, "cols": 52, "audio": 256},
        # The longest sequence (49152 tokens, 32 heads), token-exact protection: the largest pass.
        {"name": "layer_ltx_tokens", "kind": "layer", "H": 32, "frames": 16, "rows": 48, "cols": 64, "audio": 512,
         "keep_pct": 20, "protect": "tokens"},
        # Audio->video cross-attention of a saliency-update step at the longest sequence (512 audio tokens).
        {"name": "cross_ltx_update", "kind": "cross", "H": 32, "frames": 16, "rows": 48, "cols": 64, "audio": 512},
        # The same direction between updates (no score pass), odd audio length, projections in [B,N,H,d] storage.
        {"name": "cross_mid_plain_bnhd", "kind": "cross", "frames": 31, "rows": 24, "cols": 24, "audio": 157, "update": False,
         "layout": "bnhd", "keep_buffers": False},
        # The other direction of the pair: every video token attends to the audio tokens, with audio-token saliency.
        {"name": "cross_ovi_reverse", "kind": "cross", "frames": 21, "rows": 30, "cols": 52, "audio": 256, "direction": "v2a"},
        # The mask alone, rebuilt each step from fresh Q and K while the saliency is reused; [B,N,H,d] storage.
        {"name": "mask_ovi_tokens_bnhd", "kind": "mask", "frames": 21, "rows": 30, "cols": 52, "protect": "tokens",
         "layout": "bnhd"},
        # Sparse attention with short lists (10 % kept, nothing protected) and the log-sum-exp.
        {"name": "sparse_mid_keep10_lse", "kind": "sparse", "frames": 31, "rows": 24, "cols": 24, "keep_pct": 10,
         "protect_pct": 0, "lse": True},
        # Cache-reuse indicators of one block's outputs (both streams, 24 heads x 128 channels).
        {"name": "indicators_ovi", "kind": "indicators", "frames": 21, "rows": 30, "cols": 52, "audio": 256},
    ]


# Work of the largest listed pass (layer_ltx_tokens): a drawn case is kept below both.
_MAX_FLOPS = 1.1e13
_MAX_HEAD_TOKENS = 32 * 49152


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, n):
    """frames, rows, cols with a product near n (any remainder against the block size)."""
    frames = max(1, min(31, _log_int(rng, 1, max(1, min(31, n // 16)))))
    per = max(1.0, n / frames)
    rows = max(1, int(round(math.sqrt(per) * rng.uniform(0.6, 1.1))))
    return frames, rows, max(1, int(round(per / rows)))


def draw(rng: random.Random):
    kinds = ["layer"] * 5 + ["cross"] * 3 + ["mask", "sparse", "self", "indicators"]
    while True:
        d = rng.choice([128, 128, 128, 64])
        c = {"kind": rng.choice(kinds), "d": d, "B": rng.choice([1, 1, 1, 2]), "H": rng.choice([2, 4, 8, 12, 16, 24, 24, 32]),
             "layout": rng.choice(["bhnd", "bnhd"])}
        if c["kind"] == "self":
            n = _log_int(rng, 40, 512)
            c["cols"] = n
        else:
            n = _log_int(rng, 256, 49152)
            c["frames"], c["rows"], c["cols"] = _draw_grid(rng, n)
            c["audio"] = _log_int(rng, 24, 512)
        if c["kind"] in ("layer", "self", "mask", "sparse"):
            c["keep_pct"] = rng.choice([10, 20, 25, 50])
            c["protect_pct"] = rng.choice([0, 5, 5, 10, 20])
            c["protect"] = rng.choice(["blocks", "blocks", "tokens", "tokens", "cols", "sum"])
        if c["kind"] in ("layer", "cross"):
            c["update"] = rng.random() < 0.6
        if c["kind"] == "cross":
            c["direction"] = rng.choice(["a2v", "v2a"])
        if c["kind"] == "sparse":
            c["lse"] = rng.random() < 0.5
            c["protect"] = rng.choice(["blocks", "tokens"])
        c["keep_buffers"] = rng.random() < 0.7
        f = _full(c)
        if c["B"] * c["H"] * _tokens(f) <= _MAX_HEAD_TOKENS and work(c)["flops"] <= _MAX_FLOPS:
            return c


# ------------------------------------------------------------------------------------------------ inputs
def _regions(c):
    """Four sound-source regions, each about a quarter of the frames, three tenths of the rows and a fifth of the columns
    (together a little over 5 % of the tokens)."""
    f, r, w = c["frames"], c["rows"], c["cols"]
    df, dr, dw = max(1, f // 4), max(1, 3 * r // 10), max(1, w // 5)
    return tuple(((i * f) // 4, df, ((5 * i + 2) * r // 16) % max(1, r - dr + 1), dr, ((7 * i + 1) * w // 20) % max(1, w - dw + 1), dw)
                 for i in range(4))


def _workload(c):
    return wl.Workload("case", c["B"], c["H"], c["d"], c["frames"], c["rows"], c["cols"], max(1, c["audio"]), c["d"],
                       c["keep_pct"], c["protect_pct"], 1.0 if c["d"] == 128 else 0.0, _regions(c))


def _stored(x, layout):
    return x.transpose(1, 2).contiguous().transpose(1, 2) if layout == "bnhd" else x


def _saliency(c, seed, device):
    """A cached response map, fp32 [B, N]: log-normal over the tokens, raised inside the sound-source regions, summing to 1
    (what the L1-normalised scores of the steps before look like)."""
    w = _workload(c)
    n = w.n_video
    z = wl.normal_flat(seed, 11, 0, c["B"] * n, device).view(c["B"], n)
    s = torch.exp(0.3 * z + 2.0 * wl.region_mask(w, device).to(torch.float32)[None, :])
    return (s / s.sum(dim=1, keepdim=True)).contiguous()


def _counts(c):
    n, nb = _tokens(c), (_tokens(c) + c["d"] - 1) // c["d"]
    k_keep = max(1, av.avsa_count_from_percent(c["keep_pct"], nb))
    n_protect = av.avsa_count_from_percent(c["protect_pct"], nb if c["protect"] == "sum" else n)
    return k_keep, n_protect


_FLAGS = {"blocks": av.AVSA_PROTECT_ROWS, "tokens": av.AVSA_PROTECT_TOKENS,
          "cols": av.AVSA_PROTECT_ROWS | av.AVSA_PROTECT_COLS, "sum": av.AVSA_PROTECT_BLOCK_SUM | av.AVSA_PROTECT_ROWS}


def _protected_blocks(c, s):
    """bool [B, NB]: the blocks that the saliency map protects (dense rows)."""
    b, n, blk = c["B"], _tokens(c), c["d"]
    nb = (n + blk - 1) // blk
    n_protect = _counts(c)[1]
    flags = torch.zeros((b, nb * blk), dtype=torch.bool, device=s.device)
    if n_protect == 0 or c["protect"] == "tokens":
        return flags.view(b, nb, blk).any(dim=2)
    if c["protect"] == "sum":
        sums = torch.nn.functional.pad(s, (0, nb * blk - n)).view(b, nb, blk).sum(dim=2)
        return torch.zeros((b, nb), dtype=torch.bool, device=s.device).scatter_(1, sums.topk(n_protect, dim=1).indices, True)
    flags.scatter_(1, s.topk(n_protect, dim=1).indices, True)
    return flags.view(b, nb, blk).any(dim=2)


def _lists(c, q, k, s):
    """Block lists of the base pattern plus the dense rows, made with torch alone (the lists are an input here)."""
    b, h, n, d = q.shape
    nb = (n + d - 1) // d
    size = torch.full((nb,), float(d), device=q.device)
    size[-1] = float(n - (nb - 1) * d)

    def pool(x):
        x = torch.nn.functional.pad(x.float(), (0, 0, 0, nb * d - n)).view(b, h, nb, d, d).sum(dim=3)
        return x / size[:, None]

    keep = torch.zeros((b, h, nb, nb), dtype=torch.bool, device=q.device)
    keep.scatter_(3, (pool(q) @ pool(k).transpose(2, 3)).topk(_counts(c)[0], dim=3).indices, True)
    keep |= _protected_blocks(c, s)[:, None, :, None]
    where = torch.where(keep, torch.arange(nb, device=q.device), nb).sort(dim=3).values
    return torch.where(where < nb, where, -1).to(torch.int32).contiguous(), keep.sum(dim=3).to(torch.int32).contiguous()


def _bytes(n, dev):
    return torch.empty(n, dtype=torch.uint8, device=dev)


def prepare(case, seed):
    c = _full(case)
    dev = torch.device("cuda", torch.cuda.current_device())
    w = _workload(c)
    B, H, d, n, na, blk = c["B"], c["H"], c["d"], _tokens(c), c["audio"], c["d"]
    nb = (n + blk - 1) // blk
    st = {"c": c, "blk": blk}
    st["k_keep"], st["n_protect"] = _counts(c)
    if c["kind"] == "indicators":
        g = torch.Generator(device=dev).manual_seed(seed)
        for tag, rows in (("v", n), ("a", na)):
            y = torch.randn((B, rows, H * d), generator=g, device=dev)
            st["y_" + tag] = y.to(torch.bfloat16)
            st["yhat_" + tag] = (y + 0.1 * torch.randn(y.shape, generator=g, device=dev)).to(torch.bfloat16)
        st["s_cur"], st["s_anchor"] = _saliency(c, seed, dev), _saliency(c, seed + 1, dev)
        order = st["s_cur"].topk(st["n_protect"] or 1, dim=1).indices
        st["prot"] = torch.zeros((B, n), dtype=torch.uint8, device=dev).scatter_(1, order, 1)
        if c["keep_buffers"]:
            st["out"] = torch.empty((B, 8), dtype=torch.float32, device=dev)
            st["ws_i"] = _bytes(av.avsa_cache_indicators_workspace_bytes(B, n, na, H * d), dev)
        return st
    keep = c["keep_buffers"]
    if c["kind"] in ("layer", "self", "mask", "sparse"):
        q, k, v = wl.make_self_qkv(w, seed, dev)
        st["s_bar"] = _saliency(c, seed, dev)
        if c["kind"] == "sparse":
            st["col_idx"], st["col_cnt"] = _lists(c, q, k, st["s_bar"])
        st["q"], st["k"], st["v"] = (_stored(x, c["layout"]) for x in (q, k, v))
        if keep:
            if c["kind"] != "sparse":
                st["m"] = {"block_scores": torch.empty((B, H, nb, nb), dtype=torch.float32, device=dev),
                           "col_idx": torch.empty((B, H, nb, nb), dtype=torch.int32, device=dev),
                           "col_cnt": torch.empty((B, H, nb), dtype=torch.int32, device=dev),
                           "prot_tok": torch.empty((B, n), dtype=torch.uint8, device=dev),
                           "prot_blk": torch.empty((B, nb), dtype=torch.uint8, device=dev)}
                st["ws_m"] = _bytes(av.avsa_build_block_mask_workspace_bytes(B, H, n, d, blk), dev)
            st["o"] = torch.empty_strided(st["q"].shape, st["q"].stride(), dtype=torch.bfloat16, device=dev)
            st["ws_s"] = _bytes(av.avsa_sparse_self_attn_workspace_bytes(B, H, n, d, blk), dev)
            if c["lse"]:
                st["lse"] = torch.empty((B, H, n), dtype=torch.float32, device=dev)
            if c["protect"] == "tokens":
                st["ws_p"] = _bytes(av.avsa_protected_rows_attn_workspace_bytes(B, H, n, d, blk, st["n_protect"]), dev)
    if c["kind"] in ("layer", "cross"):
        qa, kc, vc = (_stored(x, c["layout"]) for x in wl.make_cross_qkv(w, seed, dev))
        # v2a swaps the roles: the video stream asks, the audio stream answers
        st["qc"], st["kc"], st["vc"] = (qa, kc, vc) if c["direction"] == "a2v" else (kc, qa, _stored(wl._tensor(w, seed, 12, na, dev), c["layout"]))
        nq, nk = st["qc"].shape[2], st["kc"].shape[2]
        st["gamma"] = 1.0 / (H * nq)
        st["cache"] = torch.full((B, nk), 1.0 / nk, dtype=torch.float32, device=dev)
        if keep:
            st["oc"] = torch.empty_strided(st["qc"].shape, st["qc"].stride(), dtype=torch.bfloat16, device=dev)
            st["lse_c"] = torch.empty((B, H, nq), dtype=torch.float32, device=dev)
            st["ws_c"] = _bytes(av.avsa_cross_attn_scores_workspace_bytes(B, H, nq, nk, d), dev)
    return st


# ------------------------------------------------------------------------------------------------ one pass
def _run_mask(st):
    c = st["c"]
    return av.avsa_build_block_mask(st["q"], st["k"], st["s_bar"] if st["n_protect"] else None, st["n_protect"], st["k_keep"],
                                    st["blk"], flags=_FLAGS[c["protect"]], out=st.get("m"), ws=st.get("ws_m"))


def _run_self(st, m):
    o, lse, _ = av.avsa_sparse_self_attn(st["q"], st["k"], st["v"], m["col_idx"], m["col_cnt"], st["blk"],
                                         want_lse=st["c"]["lse"], o=st.get("o"), lse=st.get("lse"), ws=st.get("ws_s"))
    if st["c"]["protect"] == "tokens" and "prot_tok" in m and st["n_protect"]:
        av.avsa_protected_rows_attn(st["q"], st["k"], st["v"], m["prot_tok"], st["n_protect"], st["blk"], o, lse=lse,
                                    ws=st.get("ws_p"))
    return o, lse


def _run_cross(st):
    """An update step blends the scores into the cached map in place (alpha = 0.5); other steps leave it alone."""
    if not st["c"]["update"]:
        return av.avsa_cross_attn_scores(st["qc"], st["kc"], st["vc"], want_scores=False, o=st.get("oc"), lse=st.get("lse_c"),
                                         ws=st.get("ws_c"))[:2]
    return av.avsa_cross_attn_scores(st["qc"], st["kc"], st["vc"], scores=st["cache"], score_beta=0.5,
                                     score_gamma=0.5 * st["gamma"], o=st.get("oc"), lse=st.get("lse_c"), ws=st.get("ws_c"))[:3]


def run(state):
    kind = state["c"]["kind"]
    if kind == "indicators":
        return av.avsa_cache_indicators(state["y_v"], state["yhat_v"], state["y_a"], state["yhat_a"], state["prot"], state["s_cur"],
                                        state["s_anchor"], out=state.get("out"), ws=state.get("ws_i"))[0]
    if kind == "cross":
        return _run_cross(state)
    if kind == "sparse":
        return _run_self(state, {"col_idx": state["col_idx"], "col_cnt": state["col_cnt"]})
    m = _run_mask(state)
    out = {key: m[key] for key in ("block_scores", "col_idx", "col_cnt", "prot_tok", "prot_blk")}
    if kind in ("layer", "self"):
        out["o"], out["lse"] = _run_self(state, m)
    if kind == "layer":
        out["cross"] = _run_cross(state)
    return out


# ------------------------------------------------------------------------------------------------ work and tolerance
def _pair_fraction(c):
    """Share of the (query, key) pairs that the self-attention computes: the kept blocks, and the dense rows."""
    k_keep, n_protect = _counts(c)
    n = _tokens(c)
    nb = (n + c["d"] - 1) // c["d"]
    kappa = k_keep / nb
    if c["protect"] == "tokens":
        return kappa + (0.0 if c["kind"] == "sparse" else n_protect / n)
    dense = _protected_blocks(c, _saliency(c, 0, "cpu")).float().mean().item()
    cols = dense * (1.0 - kappa) if c["protect"] == "cols" else 0.0
    return dense + (1.0 - dense) * (kappa + cols)


def work(case):
    c = _full(case)
    B, H, d, n, na = c["B"], c["H"], c["d"], _tokens(c), c["audio"]
    nb = (n + d - 1) // d
    tensor, lists, kind = 2.0 * B * H * n * d, 4.0 * B * H * nb * nb, c["kind"]
    nbytes = flops = 0.0
    if kind == "indicators":
        return {"bytes": 2.0 * B * (n + na) * H * d * 2, "flops": 6.0 * B * (n + na) * H * d}
    if kind in ("layer", "self", "mask"):          # Q and K in; block scores and lists out
        nbytes += 2 * tensor + 2 * lists + 5.0 * B * n
        flops += 2.0 * B * H * n * d + 2.0 * B * H * nb * nb * d
    if kind in ("layer", "self", "sparse"):        # Q, K, V and the lists in, O out
        nbytes += 4 * tensor + lists
        flops += 4.0 * B * H * float(n) * n * d * _pair_fraction(c)
    if kind in ("layer", "cross"):                 # the long operand pair once, the short one once; O out
        long_passes = 2.0                          # K and V of the video stream, or Q and O of it
        nbytes += long_passes * (tensor + 2.0 * B * H * na * d) + 4.0 * B * (n if c["direction"] == "a2v" else na)
        flops += (6.0 if c["update"] else 4.0) * B * H * float(n) * na * d
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "indicators":       # fp32 sums of a few million terms; the drift of Eq. 14 is a small difference from 1
        return {"rel": 1e-5, "max": 1e-5}
    if kind == "mask":             # fp32 block scores (1.4e-6 from 64 bits); a rank at a list's edge may swap with its neighbour
        return {"rel": 6e-6, "max": 2e-5, "differ": 1e-3}
    if kind in ("cross", "sparse"):    # bf16 probabilities and outputs: 2.4e-3 and 1.2e-2 from 64 bits
        return {"rel": 1e-2, "max": 0.05, "differ": 0.0}
    # the same behind a mask of its own: two blocks of nearly equal score that swap at a list's edge change their query
    # block's rows (seen once in 12288 rows against scores in 64 bits)
    return {"rel": 1e-2, "max": 0.5, "differ": 1e-3}
