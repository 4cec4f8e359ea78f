"""Kernels at the sizes where their splits can go wrong: tile edges, remainders,
the smallest and largest of their ranges. Each case is compared with the
float64 oracle (or a bit-by-bit walk) at the parity tolerances of gpu_helpers,
unless a bound is derived beside it.
"""
import numpy as np
import pytest

import oracle
from paper_2608_05780_gb300 import _binding as B
from gpu_helpers import check_lse, check_maps, check_o, np32, oracle_maps, run_cuda, to_device


def _custom(**kw):
    from test_gpu_parity import _custom as make
    return make(**kw)


# --- host ---------------------------------------------------------------------

@pytest.mark.parametrize("n_vis,tile,words,density", [
    ((), 64, 1, 0.5), ((0, 0), 64, 1, 0.5), ((1,), 64, 1, 0.5), ((64, 65, 0, 640), 64, 1, 0.1),
    ((128 * 70 + 1,), 128, 3, 0.5), ((4096,), 128, 2, 0.0), ((4096,), 128, 2, 1.0)])
def test_union_to_csr_matches_a_bit_walk(n_vis, tile, words, density):
    import torch
    rows = sum(-(-n // tile) for n in n_vis)
    rng = np.random.default_rng(3)
    bits = (rng.random((rows + 2, words, 32)) < density).astype(np.uint64)      # two spare rows, ignored
    union = (bits << np.arange(32, dtype=np.uint64)).sum(axis=2).astype(np.uint32).view(np.int32)
    row_ptr, cols = [0], []
    for r in range(rows):
        cols += [w * 32 + j for w in range(words) for j in range(32) if bits[r, w, j]]
        row_ptr.append(len(cols))
    for t in (torch.from_numpy(union), torch.from_numpy(np.asfortranarray(union))):
        got_ptr, got_cols = B.tile_union_to_csr(t, n_vis, tile)
        assert got_ptr.dtype == got_cols.dtype == np.int32
        assert got_ptr.tolist() == row_ptr and got_cols.tolist() == cols
    if rows:
        with pytest.raises(IndexError):
            B.tile_union_to_csr(torch.from_numpy(union[:rows - 1]), n_vis, tile)


# --- text sums ----------------------------------------------------------------

@pytest.mark.gpu
@pytest.mark.parametrize("n_text", [1, 31, 128, 129, 257, 400])
@pytest.mark.parametrize("tile,d,hq,hkv", [(64, 64, 6, 2), (128, 128, 7, 1)])
def test_text_sums_at_row_tile_edges(cuda_lib, n_text, tile, d, hq, hkv):
    """One text row, a full warp, a full row tile, one row more, several tiles;
    odd head groups; a last key tile of 16 columns. Inside the probe call and as
    a pass of its own."""
    probe = _custom(frames=(9, 41), n_text=(n_text, 3), hq=hq, hkv=hkv, d=d, tile=tile, window=2)
    want = oracle_maps(probe)
    for te in (False, True):
        out, ws = run_cuda(cuda_lib, probe, text_evidence=te)
        ws.free()
        check_maps([np32(out[k]) for k in ("tok", "frame", "head", "aqf")], want, probe, label=f"{n_text} rows {te}")


@pytest.mark.gpu
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("n_text", [1, 37, 129, 250])
@pytest.mark.parametrize("tile,d,hq,hkv", [(64, 64, 6, 2), (128, 128, 7, 1)])
def test_non_finite_queries_of_the_next_video_stay_there(cuda_lib, n_text, tile, d, hq, hkv, value):
    """A text tile is rounded up to 16 rows, which are the next video's first
    visual rows: their logits must not enter this video's sums. Its maps are those
    of the call with finite inputs, bit for bit."""
    import torch
    probe = _custom(frames=(9, 5), n_text=(n_text, 20), hq=hq, hkv=hkv, d=d, tile=tile, window=2)
    cut, cols = int(probe.cu_seqlens[1]), int(probe.n_vis[0])
    qkv = to_device(probe)
    bad = qkv[0].clone()
    bad[cut:] = value
    for te in (False, True):
        out, ws = run_cuda(cuda_lib, probe, qkv=qkv, text_evidence=te)
        ws.free()
        got, ws = run_cuda(cuda_lib, probe, qkv=(bad, *qkv[1:]), text_evidence=te)
        ws.free()
        frames = cols // 16
        for name, n in (("tok", cols), ("frame", frames)):
            assert torch.equal(got[name][:, :n], out[name][:, :n]), (name, te)
        assert torch.equal(got["head"][0], out["head"][0]) and torch.equal(got["aqf"][:frames], out["aqf"][:frames])


@pytest.mark.gpu
def test_evidence_overwrites_what_the_maps_held_and_accumulates_on_it(cuda_lib):
    """The overwrite and accumulate kernels on ragged sizes: NaN in the maps is
    overwritten; accumulate adds one fp32 rounding per entry."""
    import torch
    probe = _custom(frames=(3, 0, 17), n_text=(12, 40, 0), hq=6, hkv=2, d=64, tile=64, window=2)
    out, ws = run_cuda(cuda_lib, probe)
    first = [out[k] for k in ("tok", "frame", "head", "aqf")]
    dirty = [torch.full_like(m, float("nan")) for m in first]
    out, ws = run_cuda(cuda_lib, probe, ws=ws, maps=dirty)
    for a, b in zip(first, (out[k] for k in ("tok", "frame", "head", "aqf"))):
        assert torch.equal(a, b)
    base = [torch.rand_like(m) for m in first]
    out, ws = run_cuda(cuda_lib, probe, ws=ws, maps=[m.clone() for m in base], accumulate=True)
    for m0, a, b in zip(base[:2], first[:2], (out["tok"], out["frame"])):
        assert torch.equal(b, m0 + a)            # one fp32 addition per entry
    # head map and A_qf are sums of at most 17 resp. 6 non-negative frame entries
    # (and a division): fewer than 20 roundings of 2^-24
    frame = out["frame"].double()
    off = np.concatenate([[0], np.cumsum(probe.n_vis // 16)])
    head = torch.stack([frame[:, off[i]:off[i + 1]].sum(1) for i in range(3)])
    text = np.diff(probe.cu_seqlens) - probe.n_vis
    per = torch.as_tensor(np.repeat(1.0 / np.maximum(text, 1) * (text > 0), np.diff(off)) / 6, device="cuda")
    for got, want in ((out["head"], head), (out["aqf"], frame.sum(0) * per)):
        assert (got.double() - want).abs().le(20 * 2.0 ** -24 * want).all()
    ws.free()


# --- attention ----------------------------------------------------------------

def _leveled(tile, order, **kw):
    """A probe whose logits step from key tile to key tile: up or down by 8 log2
    units at every one, up by 65 in the last visual tile alone, or by 32 at tile 1
    and again at tile 21."""
    probe = _custom(**{**dict(frames=(25 * tile // kw.get("npf", 16),), n_text=(33,), hq=5, hkv=1, d=128, tile=tile,
                              window=64), **kw})
    n = int(probe.cu_seqlens[-1])
    step = np.arange(n) // tile
    if order == "one_spike":
        level = np.where(step == int(probe.n_vis[0] - 1) // tile, 4.0, 0.0)
    elif order == "two_steps":
        level = np.where(step >= 21, 4.0, np.where(step >= 1, 2.0, 0.0))
    else:
        level = 0.5 * (step if order == "rising" else step.max() - step)
    s = np.where(np.arange(128) % 3 == 0, 1.0, -1.0)
    # q . k = 128 level + noise, scale 128^-1/2: 11.3 level; bf16 values by truncation
    k = (s * level[:, None, None] + 0.0625 * probe.k).astype(np.float32)
    probe.k[:] = (k.view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32)
    probe.q[:] = s
    return probe


@pytest.mark.gpu
@pytest.mark.parametrize("tile", [64, 128])
@pytest.mark.parametrize("order", ["rising", "falling", "one_spike", "two_steps"])
def test_running_max_over_key_tiles(cuda_lib, tile, order):
    """The row maximum moves at every key tile, at none after the first, in the last
    visual tile alone, or at tile 1 and again at tile 21: the accumulator is
    rescaled at each step, at none, once, or twice with more tiles between than the
    kernel stays careful for."""
    probe = _leveled(tile, order)
    out, ws = run_cuda(cuda_lib, probe)
    ws.free()
    o_ref, lse_ref = oracle.probe(probe.q, probe.k, probe.v, probe.cu_seqlens, probe.n_vis, probe.cfg.tile,
                                  probe.row_ptr, probe.col_idx)
    check_o(np32(out["o"]), o_ref, order)
    check_lse(np32(out["lse"]), lse_ref, order)


@pytest.mark.gpu
@pytest.mark.parametrize("npf", [16, 64])
@pytest.mark.parametrize("order", ["one_spike", "two_steps"])
def test_running_max_with_cross_frame_partials(cuda_lib, order, npf):
    """The first tiles are flat, so P of a later tile's first half is formed on the
    old maximum, found too small and formed again, its partials stored twice."""
    from test_gpu_cross_frame import _check, _gpu, _oracle
    probe = _leveled(128, order, npf=npf)
    (aff, eff), (want_aff, want_eff) = _gpu(cuda_lib, probe), _oracle(probe)
    _check(aff, np.concatenate([np.asarray(x).ravel() for x in want_aff]), f"{order} A_ff")
    _check(eff, np.concatenate([np.asarray(x).ravel() for x in want_eff]), f"{order} E_ff")


@pytest.mark.gpu
@pytest.mark.parametrize("block", [16, 128])
@pytest.mark.parametrize("order", ["one_spike", "two_steps"])
def test_running_max_with_row_masks(cuda_lib, order, block):
    """As above under per-row masks that drop a third of the blocks, the masks
    applied again when P is formed again."""
    import torch
    from test_gpu_topp import _sets_from_keep
    probe = _leveled(128, order, npf=max(block, 16))
    cfg, cu, n_vis = probe.cfg, probe.cu_seqlens, probe.n_vis
    n, nv = int(cu[-1]), int(n_vis[0])
    rng = np.random.default_rng(8)
    pos = np.arange(n)
    own = np.where(pos < nv, pos // block, nv // block + (pos - nv) // block)
    blocks = nv // block + -(-(n - nv) // block)
    words = -(-blocks // 32)
    bits = rng.random((cfg.hq, words * 32, n)) < 2 / 3
    ids = np.arange(words * 32)[:, None]
    bits = (bits & (ids < own)) | (ids == own)
    bits[:, 0] |= rng.random((cfg.hq, n)) < 0.9      # the first block mostly kept: a flat first tile
    packed = (bits.reshape(cfg.hq, words, 32, n).astype(np.uint64) << np.arange(32, dtype=np.uint64)[:, None]).sum(2)
    keep = torch.from_numpy(packed.astype(np.uint32).view(np.int32)).cuda()
    q, k, v = to_device(probe)
    o, lse, ws = cuda_lib.evisel_probe_attention(q, k, v, cu, n_vis, cfg.tokens_per_frame, cfg.tile, probe.row_ptr,
                                                 probe.col_idx, keep=keep, keep_block=block)
    torch.cuda.synchronize()
    assert cuda_lib.evisel_status(ws) == 0
    ws.free()
    rows = np.unique(np.concatenate([rng.integers(0, n, 60), np.arange(n - 40, n)]))
    kept = _sets_from_keep(keep, np.arange(n), cu, n_vis, block)
    o_ref, lse_ref = oracle.probe_rows_topp(probe.q, probe.k, probe.v, cu, n_vis, block, kept, rows)
    check_o(np32(o)[rows], o_ref, order)
    check_lse(np32(lse)[:, rows], lse_ref, order)


# --- top-p masks, masked text sums, coarse map ---------------------------------

TOPP = {   # heads per KV group: four at a time, then the rest; ragged tiles and text blocks
    "group5_b16_d64_t64": (dict(frames=(21, 0, 5), n_text=(29, 7, 0), hq=10, hkv=2, d=64, tile=64, window=2), 16),
    "group9_b32_d128_t128": (dict(frames=(19,), n_text=(130,), npf=32, hq=9, hkv=1, d=128, tile=128, window=2), 32),
    "mha_b64_t64": (dict(frames=(12, 9), n_text=(65, 1), npf=64, hq=3, hkv=3, d=128, tile=64, window=2), 64),
    "group7_b128_t128": (dict(frames=(9,), n_text=(200,), npf=128, hq=7, hkv=1, d=128, tile=128, window=2), 128),
    "b16_past_512_blocks": (dict(frames=(530,), n_text=(20,), hq=4, hkv=1, d=64, tile=128, window=2), 16),
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(TOPP))
def test_topp_chain_at_edges(cuda_lib, name):
    """Retained sets (and their tile union) by the rule's properties, then on
    these sets the probe's evidence and the coarse map against the oracle."""
    import torch
    from test_gpu_topp import _check_sets, _logit_bounds, _sets_from_keep
    kw, block = TOPP[name]
    tau = 0.8
    probe = _custom(**kw)
    cfg, cu, n_vis = probe.cfg, probe.cu_seqlens, probe.n_vis
    n = int(cu[-1])
    q, k, v = to_device(probe)
    keep, uni, ws = cuda_lib.evisel_topp_mask(q, k, cu, n_vis, cfg.tokens_per_frame, cfg.tile, block, tau)
    coarse = cuda_lib.evisel_coarse_evidence(q, k, cu, n_vis, cfg.tokens_per_frame, cfg.tile, block, keep, ws)
    torch.cuda.synchronize()
    rng = np.random.default_rng(1)
    rows = np.unique(np.concatenate([cu[:-1], cu[1:] - 1, rng.integers(0, n, 20)]))
    rows = rows[(rows >= 0) & (rows < n)]
    bits = keep[:, :, torch.as_tensor(rows, device="cuda")].cpu().numpy().view(np.uint32)
    sets = {(h, int(row)): [w * 32 + j for w in range(bits.shape[1]) for j in range(32) if bits[h, w, r] >> j & 1]
            for h in range(bits.shape[0]) for r, row in enumerate(rows)}
    _, probs = oracle.retained_blocks(probe.q, probe.k, cu, n_vis, block, tau, rows=rows)
    _check_sets(sets, probs, _logit_bounds(probe.q, probe.k, cu, n_vis, block, rows), cu, n_vis, block, tau, name)
    # the union, bit for bit, from the masks
    row_ptr, col_idx = B.tile_union_to_csr(uni, n_vis, cfg.tile)
    all_bits = keep.cpu().numpy().view(np.uint32)
    r = 0
    for b, nv in enumerate(n_vis):
        for t in range(-(-int(nv) // cfg.tile)):
            span = all_bits[:, :, int(cu[b]) + t * cfg.tile:int(cu[b]) + min((t + 1) * cfg.tile, int(nv))]
            words = np.bitwise_or.reduce(np.bitwise_or.reduce(span, axis=2), axis=0)
            ids = np.nonzero(np.unpackbits(words.view(np.uint8), bitorder="little"))[0]
            assert col_idx[row_ptr[r]:row_ptr[r + 1]].tolist() == sorted(set((ids * block // cfg.tile).tolist())), (b, t)
            r += 1
    text = np.concatenate([np.arange(int(cu[b]) + int(n_vis[b]), int(cu[b + 1])) for b in range(len(n_vis))])
    kept = _sets_from_keep(keep, text, cu, n_vis, block)
    want = oracle.coarse_evidence(probe.q, probe.k, cu, n_vis, cfg.tokens_per_frame, block, kept)
    check_maps([np32(m) for m in coarse], list(want), probe, label=f"{name} coarse")
    o, lse, ws = cuda_lib.evisel_probe_attention(q, k, v, cu, n_vis, cfg.tokens_per_frame, cfg.tile, row_ptr, col_idx,
                                                 ws=ws, keep=keep, keep_block=block)
    maps = cuda_lib.evisel_evidence_reduce(ws, cfg.hq, n_vis, cfg.tokens_per_frame, len(n_vis))
    torch.cuda.synchronize()
    assert cuda_lib.evisel_status(ws) == 0
    want = oracle.evidence_topp(probe.q, probe.k, cu, n_vis, cfg.tokens_per_frame, block, kept)
    check_maps([np32(m) for m in maps], list(want), probe, label=f"{name} masked evidence")
    ws.free()


@pytest.mark.gpu
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("name", ["group5_b16_d64_t64", "group9_b32_d128_t128"])
def test_non_finite_keys_that_no_text_row_keeps_add_nothing(cuda_lib, name, value):
    """After a masked probe a block that no text row keeps adds 0 to the maps
    whatever its keys hold: the maps are those of finite keys, bit for bit. A
    non-finite text query likewise adds nothing to the blocks its row drops, where
    other rows' sums stand."""
    import torch
    kw, block = TOPP[name]
    probe = _custom(**kw)
    cfg, cu, n_vis = probe.cfg, probe.cu_seqlens, probe.n_vis
    q, k, v = to_device(probe)
    keep, uni, ws = cuda_lib.evisel_topp_mask(q, k, cu, n_vis, cfg.tokens_per_frame, cfg.tile, block, 0.3)
    row_ptr, col_idx = B.tile_union_to_csr(uni, n_vis, cfg.tile)
    nv, end = int(n_vis[0]), int(cu[1])
    victims = [1, nv // block - 1]               # blocks of the first video, dropped from its text rows
    for j in victims:
        keep[:, j >> 5, nv:end] &= ~(1 << (j & 31))

    def maps(keys, q=q):
        w = cuda_lib.Workspace()
        cuda_lib.evisel_probe_attention(q, keys, v, cu, n_vis, cfg.tokens_per_frame, cfg.tile, row_ptr, col_idx, ws=w,
                                        keep=keep, keep_block=block)
        out = cuda_lib.evisel_evidence_reduce(w, cfg.hq, n_vis, cfg.tokens_per_frame, len(n_vis))
        torch.cuda.synchronize()
        assert cuda_lib.evisel_status(w) == 0
        w.free()
        return out
    bad = k.clone()
    for j in victims:
        bad[j * block:(j + 1) * block] = value
    want, got = maps(k), maps(bad)
    for j in victims:
        assert (want[0][:, j * block:(j + 1) * block] == 0).all()
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    for j in victims:                            # kept by the second text row alone
        keep[:, j >> 5, nv + 1] |= 1 << (j & 31)
    bad = q.clone()
    bad[nv] = value
    want, got = maps(k)[0], maps(k, bad)[0]
    # one pair per key, its logit summed over d in another order: 2 d 2^-24 sum |q k| scale
    # below 2 * 128 * 2^-24 * 400 / sqrt(64) = 8e-4 (sum |q k| < 400 asserted)
    assert (q[nv + 1].float().norm(dim=-1).max() * k[:nv].float().norm(dim=-1).max()).item() < 400
    for j in victims:
        a, b = (m[:, j * block:(j + 1) * block] for m in (want, got))
        assert (a > 0).all() and ((b - a).abs() <= 8e-4 * a).all()
    ws.free()


@pytest.mark.gpu
def test_coarse_map_takes_a_million_text_rows(cuda_lib):
    """2,048 videos of one frame and 512 text rows, all alike: 67,584 groups of 16
    text rows, more than a grid holds in y. Every video's maps are bit for bit
    those of the call on one of them."""
    import torch
    n_text, copies = 512, 2048
    probe = _custom(frames=(1,), n_text=(n_text,), hq=1, hkv=1, d=64, tile=64, window=2)
    one = to_device(probe)[:2]
    n = int(probe.cu_seqlens[-1])

    def maps(videos):
        q, k = (t.repeat(videos, 1, 1) for t in one)
        cu, n_vis = np.arange(videos + 1, dtype=np.int32) * n, np.full(videos, n - n_text, np.int32)
        keep, _, ws = cuda_lib.evisel_topp_mask(q, k, cu, n_vis, 16, 64, 16, 0.9, union=False)
        out = cuda_lib.evisel_coarse_evidence(q, k, cu, n_vis, 16, 64, 16, keep, ws)
        torch.cuda.synchronize()
        assert cuda_lib.evisel_status(ws) == 0
        ws.free()
        return out
    want = maps(1)
    assert (want[0] > 0).all()
    for name, a, b in zip(("tok", "frame", "head", "aqf"), want, maps(copies)):
        assert torch.equal(b, a.repeat(copies, 1) if name == "head" else a.repeat(*[1] * (a.dim() - 1), copies)), name


@pytest.mark.gpu
def test_coarse_map_finds_every_videos_rows_and_blocks(cuda_lib):
    """300 videos with 0 to 40 blocks and 0 to 40 text rows: groups of 32 blocks
    and of 8 and 16 rows, partial and empty ones among them, each found by
    bisection. Every video's maps are bit for bit those of a call on it alone."""
    import torch
    rng = np.random.default_rng(5)
    frames, text = rng.integers(0, 41, 300), rng.integers(0, 41, 300)
    frames[[0, 7, 8, 299]] = text[[0, 8, 9, 299]] = 0
    frames[20], text[20] = 70, 129               # more than one group of each
    n_vis = (16 * frames).astype(np.int32)
    cu = np.concatenate([[0], np.cumsum(n_vis + text)]).astype(np.int32)
    g = torch.Generator(device="cuda").manual_seed(6)
    q, k = (torch.randn(int(cu[-1]), h, 64, device="cuda", generator=g).bfloat16() for h in (4, 2))

    def maps(q, k, cu, n_vis):
        keep, _, ws = cuda_lib.evisel_topp_mask(q, k, cu, n_vis, 16, 64, 16, 0.9, union=False)
        out = cuda_lib.evisel_coarse_evidence(q, k, cu, n_vis, 16, 64, 16, keep, ws)
        torch.cuda.synchronize()
        assert cuda_lib.evisel_status(ws) == 0
        ws.free()
        return out
    tok, frame, head, aqf = maps(q, k, cu, n_vis)
    vis, fr = np.concatenate([[0], np.cumsum(n_vis)]), np.concatenate([[0], np.cumsum(frames)])
    for b in [0, 1, 6, 7, 8, 9, 10, 19, 20, 21, 298, 299, *range(30, 290, 13)]:
        if cu[b] == cu[b + 1]:
            assert (head[b] == 0).all()
            continue
        a, e = int(cu[b]), int(cu[b + 1])
        one = maps(q[a:e].contiguous(), k[a:e].contiguous(), np.array([0, e - a], np.int32), n_vis[b:b + 1])
        got = (tok[:, vis[b]:vis[b + 1]], frame[:, fr[b]:fr[b + 1]], head[b:b + 1], aqf[fr[b]:fr[b + 1]])
        for x, y in zip(one, got):
            assert torch.equal(x, y), b


# --- plans --------------------------------------------------------------------

@pytest.mark.gpu
def test_a_changed_mask_is_replanned_and_an_invalid_one_still_refused(cuda_lib):
    """The plan's description is compared by value in the caller's arrays: one
    changed in place is planned anew, and refused if it is not valid."""
    import torch
    probe = _custom(frames=(40,), n_text=(20,), hq=4, hkv=2, d=64, tile=64, window=2, extra=3)
    full = _custom(frames=(40,), n_text=(20,), hq=4, hkv=2, d=64, tile=64, window=40)
    q, k, v = to_device(probe)

    def call(ws, row_ptr, col_idx):
        cfg = probe.cfg
        return cuda_lib.evisel_probe_attention(q, k, v, probe.cu_seqlens, probe.n_vis, cfg.tokens_per_frame, cfg.tile,
                                               row_ptr, col_idx, ws=ws)
    row_ptr, col_idx = probe.row_ptr.copy(), probe.col_idx.copy()
    o, lse, ws = call(None, row_ptr, col_idx)
    first = o.clone()
    # in place: the last row tile keeps other tiles (same counts, so only the ids differ)
    r = len(row_ptr) - 2
    a, b = int(row_ptr[r]), int(row_ptr[r + 1])
    free = [c for c in range(r) if c not in col_idx[a:b]]
    assert free and b - a >= 2
    saved = col_idx[a:b].copy()
    col_idx[a:b] = np.sort(np.concatenate([[free[0]], saved[1:]]))
    o2, _, ws = call(ws, row_ptr, col_idx)
    fresh, _, ws2 = call(None, row_ptr, col_idx)
    assert torch.equal(o2, fresh) and not torch.equal(o2, first)
    for bad in (-1, r + 1):                      # out of range; after the row tile
        broken = col_idx.copy()
        broken[b - 1 if bad > 0 else a] = bad
        with pytest.raises(B.EviselError):
            call(ws, row_ptr, broken)
    o3, _, ws = call(ws, full.row_ptr, full.col_idx)
    fresh3, _, ws2 = call(ws2, full.row_ptr, full.col_idx)
    assert torch.equal(o3, fresh3)
    ws.free()
    ws2.free()
