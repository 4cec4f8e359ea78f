"""Performance cases of the sparse-prefill evidence probe, through the package's public entry points.

A case is one call, or the few calls in a row, that a program makes per transformer layer:

  step     evisel_probe_attention + evisel_evidence_reduce over the packed videos (``layers`` of them, the
           evidence maps summed over the layers), with the text-row probabilities read back from the
           probe's spill (evidence = "spill", the default) or formed again ("recompute")
  noalloc  the same step through the entry point that allocates nothing, with its default status read
  cues     every cue of one layer: the probe with cross-frame partials, the text-row maps, A_if, A_ff, E_ff
  retain   the top-p mask builder alone
  sparse   the whole sparse prefill of one layer: builder, host CSR of the union, the probe restricted to
           each row's retained blocks, the evidence maps
  coarse   the evidence of the coarse token-level map on retained sets that are there already

Inputs are drawn on the GPU with the recipes of the package's workloads: "iid" Q/K/V ~ N(0,1)/sqrt(d) with 5%
of the frames planted towards the query, "unit" N(0,1) (logits of unit scale), "sharp" 4 N(0,1) for Q and K
(logits of a standard deviation near 16: the running maximum moves), "clustered" block topics with queries
aimed at a few earlier blocks (attention concentrated on a small share of the history).
"""
import math

import numpy as np
import torch

import paper_2608_05780_gb300 as ev

BF16 = torch.bfloat16


# ---------------------------------------------------------------- cases
def _case(name, kind, frames, text, npf, heads, d, tile, window, extra=0, regime="iid", layers=1,
          evidence="spill", block=64, tau=0.97, buffers="kept"):
    c = dict(kind=kind, frames=frames, text=text, npf=npf, hq=heads[0], hkv=heads[1], d=d, tile=tile,
             window=window, extra=extra, regime=regime, layers=layers, evidence=evidence, block=block, tau=tau,
             buffers=buffers)
    if name:
        c["name"] = name
    return c


QWEN = (28, 4)          # query / KV heads of the 7B model whose attention shapes the workloads have

# Frames and query lengths of the packed 8-video batch (512-2048 frames, 64-256 text tokens a video).
_BATCH8_FRAMES = "1628,1961,1866,1297,1957,2012,2003,636"
_BATCH8_TEXT = "151,181,118,136,185,218,176,97"


def listed():
    return [
        # The smallest clip (32 frames of 16 tokens, 64-token tiles, d = 64): launches and host time are
        # what it costs. Called the shortest way: the calls allocate their outputs, the workspace is kept.
        _case("tiny_step", "step", "32", "32", 16, (4, 2), 64, 64, 2, buffers="new"),
        # A short clip in a server that lets the library allocate nothing; waits for the status, as by default.
        _case("noalloc_clip", "noalloc", "96", "45", 16, QWEN, 128, 128, 4),
        # One layer of a four-minute clip (4,160 tokens): the ordinary small request.
        _case("single_step", "step", "256", "64", 16, QWEN, 128, 128, 4),
        # Ragged packed requests: odd frame counts, small frames, short last tiles, a query of one token and
        # one over several tiles, 64-token tiles with d = 128, logits sharp enough to move the running maximum.
        _case("ragged_batch", "step", "333,57,1,190,461", "37,1,200,64,129", 8, (16, 8), 128, 64, 3, extra=3,
              regime="sharp", evidence="recompute"),
        # A probe over the depth of a model: four layers of a 16,512-token video, maps summed over the layers.
        _case("depth_layers", "step", "1024", "128", 16, QWEN, 128, 128, 8, layers=4),
        # The benchmark's headline: a long video, 65,664 tokens, window plus far tiles, default evidence.
        _case("long65k_step", "step", "1024", "128", 64, QWEN, 128, 128, 16, extra=32),
        # The largest batch: 8 videos, 215 thousand tokens, with the evidence mode that needs no spill.
        _case("batch8_recompute", "step", _BATCH8_FRAMES, _BATCH8_TEXT, 16, QWEN, 128, 128, 8,
              evidence="recompute"),
        # Everything the selector reads of one layer of a 24,704-token video: A_qf's maps, A_if, A_ff and E_ff.
        _case("cues_24k", "cues", "384", "128", 64, QWEN, 128, 128, 16, extra=32),
        # The same cues of a short clip with small frames.
        _case("cues_4k", "cues", "251", "70", 16, QWEN, 128, 128, 4),
        # The mask builder on a long video in the regime that top-p retention is made for.
        _case("retain_65k", "retain", "1024", "128", 64, QWEN, 128, 128, 16, regime="clustered"),
        # A sparse prefill layer from the keys to the maps on a 24,704-token video.
        _case("sparse_24k", "sparse", "384", "128", 64, QWEN, 128, 128, 16, regime="clustered"),
        # The coarse map's evidence for a 16-thousand-token video with near-uniform attention.
        _case("coarse_16k", "coarse", "509", "100", 32, QWEN, 128, 128, 8, regime="unit", block=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# The most visual tokens of a drawn case, per kind (a case costs no more than the largest listed one).
_MAX_VIS = dict(step=60000, noalloc=6000, cues=32000, retain=60000, sparse=24000, coarse=40000)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "noalloc", "cues", "cues", "retain", "sparse", "coarse"])
    evidence = rng.choice(["spill", "recompute"]) if kind in ("step", "noalloc") else "spill"
    heads, d = rng.choice([(QWEN, 128), (QWEN, 128), ((16, 8), 128), ((4, 2), 64), ((32, 8), 128), ((6, 2), 64)])
    tile = rng.choice([128, 128, 64])
    sizes = [n for n in (8, 16, 32, 64) if n <= tile and (n >= 16 or kind in ("step", "noalloc"))]
    npf = rng.choice(sizes)
    cap = _MAX_VIS[kind]
    if kind == "step" and evidence == "recompute":
        cap = 160000
    total = _log_int(rng, 512, cap)
    n_videos = 1 if total < 2048 else rng.choice([1, 1, 2, 3, 5])
    weights = [rng.uniform(0.3, 1.7) for _ in range(n_videos)]
    frames = [max(1, int(total * w / sum(weights)) // npf) for w in weights]
    text = [rng.randint(8, 256) for _ in range(n_videos)]
    if kind == "noalloc" and heads[0] * sum(n * npf * (t + 31) for n, t in zip(frames, text)) * 4 > 40 << 20:
        evidence = "recompute"          # the spill would not fit the fixed scratch
    regime = rng.choice(["iid", "iid", "unit", "sharp"]) if kind in ("step", "noalloc", "cues") else \
        rng.choice(["clustered", "clustered", "unit"])
    return _case(None, kind, ",".join(map(str, frames)), ",".join(map(str, text)), npf, heads, d, tile,
                 window=rng.randint(2, 16), extra=rng.choice([0, 0, 8, 32]) if kind in ("step", "cues") else 0,
                 regime=regime, layers=rng.choice([1, 1, 2]) if kind == "step" and total < 20000 else 1,
                 evidence=evidence, block=rng.choice([b for b in (16, 32, 64) if b <= npf] or [16]),
                 tau=rng.choice([0.9, 0.97]), buffers=rng.choice(["kept", "new"]))


# ---------------------------------------------------------------- inputs
def _shape(case):
    frames = [int(x) for x in case["frames"].split(",")]
    text = [int(x) for x in case["text"].split(",")]
    n_vis = np.array([f * case["npf"] for f in frames], np.int32)
    cu = np.zeros(len(frames) + 1, np.int32)
    cu[1:] = np.cumsum(n_vis + np.array(text))
    return frames, text, n_vis, cu


def _mask(case, seed):
    """CSR of the tile mask: the sink tile, a causal window, and ``extra`` random earlier tiles per row tile."""
    _, _, n_vis, _ = _shape(case)
    rng = np.random.default_rng([seed, 1])
    row_ptr, cols = [0], []
    for nv in n_vis:
        for r in range(-(-int(nv) // case["tile"])):
            lo = max(0, r - case["window"] + 1)
            kept = [0] if lo > 0 else []
            if case["extra"] and lo > 1:
                kept += sorted(1 + rng.permutation(lo - 1)[:case["extra"]])
            cols.extend(kept)
            cols.extend(range(lo, r + 1))
            row_ptr.append(len(cols))
    return np.array(row_ptr, np.int32), np.array(cols, np.int32)


def _inputs(case, seed, layer=0):
    """Q, K and V of one layer on the GPU (bf16), drawn from the seed."""
    frames, text, n_vis, cu = _shape(case)
    n, hq, hkv, d = int(cu[-1]), case["hq"], case["hkv"], case["d"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed((seed * 131 + layer) & 0x7FFFFFFFFFFF)
    dev = dict(device="cuda", generator=gen)
    div = math.sqrt(d) if case["regime"] == "iid" else 1.0
    gain = 4.0 if case["regime"] == "sharp" else 1.0
    q = torch.randn((n, hq, d), **dev) * (gain / div)
    k = torch.randn((n, hkv, d), **dev) * (gain / div)
    v = torch.randn((n, hkv, d), **dev) / div
    rng = np.random.default_rng([seed, 2])
    gq = hq // hkv
    for b, (f, t) in enumerate(zip(frames, text)):
        s, nv, npf = int(cu[b]), int(n_vis[b]), case["npf"]
        if case["regime"] == "iid":
            mean_q = q[s + nv:s + nv + t].reshape(t, hkv, gq, d).mean((0, 2))
            pick = torch.from_numpy(rng.choice(f, max(1, f // 20), replace=False)).cuda()
            k[s:s + nv].view(f, npf, hkv, d)[pick] += 2.0 * mean_q
        elif case["regime"] == "clustered":
            n_blk = f + -(-t // npf)
            topic = torch.randn((n_blk, hkv, d), **dev)
            blk = torch.cat([torch.arange(nv, device="cuda") // npf, f + torch.arange(t, device="cuda") // npf])
            k[s:s + nv + t] += 3.0 * topic[blk]
            starts = list(range(0, nv, case["tile"])) + [nv + a for a in range(0, t, case["tile"])]
            want, weight = np.zeros((len(starts), 8), np.int64), np.zeros((len(starts), 8), np.float32)
            for i, a in enumerate(starts):
                hist = a // npf if a < nv else f + (a - nv) // npf    # blocks that end before the tile
                ids = list(range(max(0, hist - 4), hist))
                ids += list(rng.integers(0, hist - 4, 4)) if hist > 4 else []
                want[i, :len(ids)], weight[i, :len(ids)] = ids, 1.0 / math.sqrt(max(1, len(ids)))
            centre = (topic[torch.from_numpy(want).cuda()] * torch.from_numpy(weight).cuda()[..., None, None]).sum(1)
            row_tile = torch.cat([torch.arange(nv, device="cuda") // case["tile"],
                                  -(-nv // case["tile"]) + torch.arange(t, device="cuda") // case["tile"]])
            q[s:s + nv + t] = 0.25 * q[s:s + nv + t] + centre.repeat_interleave(gq, 1)[row_tile]
    return q.to(BF16), k.to(BF16), v.to(BF16)


# ---------------------------------------------------------------- a program's state and its pass
def prepare(case, seed):
    frames, text, n_vis, cu = _shape(case)
    hq, npf, n_videos = case["hq"], case["npf"], len(frames)
    n, total_vis, total_frames = int(cu[-1]), int(n_vis.sum()), sum(frames)
    s = dict(case=case, cu=cu, n_vis=n_vis, ws=ev.Workspace(),
             layers=[_inputs(case, seed, i) for i in range(case["layers"])])
    if case["kind"] in ("step", "noalloc", "cues"):
        s["mask"] = _mask(case, seed)
    f32 = dict(dtype=torch.float32, device="cuda")
    s["maps"] = {}
    s["outs"] = [{} for _ in range(case["layers"])]
    if case["buffers"] == "kept" or case["kind"] == "noalloc":
        s["maps"] = dict(tok=torch.empty((hq, total_vis), **f32), frame=torch.empty((hq, total_frames), **f32),
                         head=torch.empty((n_videos, hq), **f32), aqf=torch.empty((total_frames,), **f32))
        if case["kind"] not in ("retain", "coarse"):
            s["outs"] = [dict(o=torch.empty((n, hq, case["d"]), dtype=BF16, device="cuda"),
                              lse=torch.empty((hq, n), **f32)) for _ in range(case["layers"])]
    if case["kind"] == "cues" and case["buffers"] == "kept":
        s["aif"] = torch.empty((total_frames, npf, npf), **f32)
        s["aff"] = torch.empty((sum((f - 1) ** 2 for f in frames),), **f32)
        s["eff"] = torch.empty((total_frames,), **f32)
    if case["kind"] == "coarse":
        q, k, _ = s["layers"][0]
        s["keep"], _, _ = ev.evisel_topp_mask(q, k, cu, n_vis, npf, case["tile"], case["block"], case["tau"],
                                              ws=s["ws"], union=False)
    return s


def run(state):
    case = state["case"]
    return {"step": _run_step, "noalloc": _run_noalloc, "cues": _run_cues, "retain": _run_retain,
            "sparse": _run_sparse, "coarse": _run_coarse}[case["kind"]](state, case)


def _run_step(s, c):
    shape = (s["cu"], s["n_vis"], c["npf"], c["tile"], *s["mask"])
    outs, maps = [], s["maps"]
    for i, qkv in enumerate(s["layers"]):
        o, lse, _ = ev.evisel_probe_attention(*qkv, *shape, ws=s["ws"], text_evidence=c["evidence"] == "recompute",
                                              **s["outs"][i])
        got = ev.evisel_evidence_reduce(s["ws"], c["hq"], s["n_vis"], c["npf"], len(s["n_vis"]),
                                        accumulate=i > 0, **maps)
        maps = dict(zip(("tok", "frame", "head", "aqf"), got))
        outs.append((o, lse))
    return {"layers": outs, "maps": list(got)}


def _run_noalloc(s, c):
    o, lse = s["outs"][0]["o"], s["outs"][0]["lse"]
    status = ev.evisel_probe_evidence_noalloc(*s["layers"][0], s["cu"], s["n_vis"], c["npf"], c["tile"], *s["mask"],
                                              o, lse, **s["maps"], text_evidence=c["evidence"] == "recompute")
    return {"layers": [(o, lse)], "maps": list(s["maps"].values()), "status": status}


def _run_cues(s, c):
    args = (*s["layers"][0], s["cu"], s["n_vis"], c["npf"], c["tile"], *s["mask"])
    o, lse, ws = ev.evisel_probe_attention(*args, ws=s["ws"], cross_frame=True, **s["outs"][0])
    maps = ev.evisel_evidence_reduce(ws, c["hq"], s["n_vis"], c["npf"], len(s["n_vis"]), **s["maps"])
    aif = ev.evisel_intra_frame_evidence(*args, o, lse, ws, aif=s.get("aif"))
    aff, eff = ev.evisel_cross_frame_evidence(*args, o, lse, ws, aff=s.get("aff"), eff=s.get("eff"))
    return {"layers": [(o, lse)], "maps": list(maps), "aif": aif, "aff": aff, "eff": eff}


def _builder(s, c, **kw):
    q, k, _ = s["layers"][0]
    return ev.evisel_topp_mask(q, k, s["cu"], s["n_vis"], c["npf"], c["tile"], c["block"], c["tau"], ws=s["ws"], **kw)


def _run_retain(s, c):
    keep, union, _ = _builder(s, c)
    return {"keep": keep, "union": union}


def _run_sparse(s, c):
    keep, union, ws = _builder(s, c)
    row_ptr, col_idx = ev.tile_union_to_csr(union, s["n_vis"], c["tile"])
    o, lse, _ = ev.evisel_probe_attention(*s["layers"][0], s["cu"], s["n_vis"], c["npf"], c["tile"], row_ptr, col_idx,
                                          ws=ws, keep=keep, keep_block=c["block"], **s["outs"][0])
    maps = ev.evisel_evidence_reduce(ws, c["hq"], s["n_vis"], c["npf"], len(s["n_vis"]), **s["maps"])
    return {"keep": keep, "union": union, "layers": [(o, lse)], "maps": list(maps)}


def _run_coarse(s, c):
    q, k, _ = s["layers"][0]
    return {"maps": list(ev.evisel_coarse_evidence(q, k, s["cu"], s["n_vis"], c["npf"], c["tile"], c["block"],
                                                   s["keep"], s["ws"], **s["maps"]))}


# ---------------------------------------------------------------- what a pass cannot do without
def _pairs(case):
    """(query, key) pairs per head that the masks of the probe keep, and the text rows' visual pairs."""
    frames, text, n_vis, _ = _shape(case)
    row_ptr, cols = _mask(case, 0)
    tile, pairs, text_pairs, r = case["tile"], 0, 0, 0
    for nv, t in zip((int(x) for x in n_vis), text):
        for i in range(-(-nv // tile)):
            rows = min(tile, nv - i * tile)
            kept = cols[row_ptr[r]:row_ptr[r + 1]]
            pairs += rows * tile * (len(kept) - 1) + rows * (rows + 1) // 2
            r += 1
        text_pairs += t * nv
        pairs += t * nv + t * (t + 1) // 2
    return pairs, text_pairs


def work(case):
    frames, text, n_vis, cu = _shape(case)
    hq, hkv, d, npf, block = case["hq"], case["hkv"], case["d"], case["npf"], case["block"]
    n, vis, tot_f = int(cu[-1]), int(n_vis.sum()), sum(frames)
    q_b, kv_b, out_b = 2 * n * hq * d, 2 * n * hkv * d, 2 * n * hq * d + 4 * n * hq
    maps_b = 4 * (hq * vis + hq * tot_f + len(frames) * hq + tot_f)
    n_blk = [int(v) // block + -(-t // block) for v, t in zip(n_vis, text)]
    keep_b = 4 * hq * n * -(-max(n_blk) // 32)
    # the builder: one q . k_bar product per (head, row, block that ends before it)
    build_f = sum(2.0 * d * hq * (int(v) + t) * nb / 2 for v, t, nb in zip(n_vis, text, n_blk)) + 2.0 * n * hkv * d
    if case["kind"] == "retain":
        return {"bytes": q_b + kv_b + keep_b, "flops": build_f}
    if case["kind"] == "coarse":
        text_n = sum(text)
        kbar_b = 2 * sum(n_blk) * hkv * d
        flops = sum(2.0 * d * hq * t * nb for t, nb in zip(text, n_blk))
        return {"bytes": 2 * text_n * (hq + hkv) * d + kbar_b + 4 * hq * text_n * max(n_blk) // 32 + maps_b,
                "flops": flops}
    if case["kind"] == "sparse":
        # clustered rows hold their mass in about eight blocks and the row's own one
        pairs = sum(int(v) + t for v, t in zip(n_vis, text)) * 9 * block
        return {"bytes": q_b + 2 * kv_b + keep_b + out_b + maps_b, "flops": build_f + 4.0 * d * hq * pairs}
    pairs, text_pairs = _pairs(case)
    flops = 4.0 * d * hq * pairs
    size = q_b + 2 * kv_b + out_b + maps_b
    if case["kind"] == "cues":
        size += 4 * (tot_f * npf * npf + sum((f - 1) ** 2 for f in frames) + tot_f)
    return {"bytes": size * case["layers"], "flops": flops * case["layers"]}


def tolerance(case):
    # O is bf16 (2^-9 relative rounding) and P is rounded to bf16 before P.V: the results are 1.4e-3 to 1.8e-3 off
    # the 64-bit ones in O and 5e-8 to 3e-6 in the fp32 outputs. One bf16 step of a value is 2^-8 of it.
    # Retained sets: blocks within 2^-14 of a row's logit range count as ties, so that a set ordered by the exact
    # logits (from the same bf16 block means) differs in 1e-5 to 4e-4 of the bit words. Where sets are drawn in
    # the pass or before it, such a row moves the maps: 3e-4 of the coarse maps in all, and a token's entry by up
    # to the share that one text row has in it.
    if case["kind"] == "retain":
        return {"rel": 0.0, "differ": 1.6e-3}
    if case["kind"] == "sparse":
        return {"rel": 1e-2, "max": 0.25, "differ": 1.6e-3}
    if case["kind"] == "coarse":
        return {"rel": 1.2e-3, "max": 0.25}
    return {"rel": 8e-3, "max": 0.08}


# ---------------------------------------------------------------- the same in 64 bits
def _sets(q, k, case, b, shape):
    """Top-p sets of video b in 64 bits: bool [hq, rows, blocks], with the rows' own blocks."""
    frames, text, n_vis, cu = shape
    s, nv, t, B = int(cu[b]), int(n_vis[b]), text[b], case["block"]
    hq, hkv, d, n = case["hq"], case["hkv"], case["d"], nv + t
    nvb, nb = nv // B, nv // B + -(-t // B)
    kd = k[s:s + n].double()
    kbar = torch.empty((nb, hkv, d), dtype=torch.float64, device="cuda")
    if nvb:
        kbar[:nvb] = kd[:nv].view(nvb, B, hkv, d).mean(1)
    for j in range(nvb, nb):
        kbar[j] = kd[nv + (j - nvb) * B:nv + (j - nvb + 1) * B].mean(0)
    pos = torch.arange(n, device="cuda")
    own = torch.where(pos < nv, pos // B, nvb + (pos - nv) // B)
    ids = torch.arange(nb, device="cuda")
    keep = torch.zeros((hq, n, nb), dtype=torch.bool, device="cuda")
    for h in range(hq):
        g = (q[s:s + n, h].double() @ kbar[:, h // (hq // hkv)].T) / math.sqrt(d)
        g = g.masked_fill(ids[None] >= own[:, None], -math.inf)
        p = torch.softmax(g, 1).nan_to_num(0.0)
        order = torch.sort(p, dim=1, descending=True, stable=True)
        before = torch.cumsum(order.values, 1) - order.values
        keep[h].scatter_(1, order.indices, before < case["tau"])
        keep[h] &= ids[None] < own[:, None]
        keep[h, pos, own] = True
    return keep, kbar, own


def _exact_layer(case, seed, layer, mask):
    """O, LSE, token map, A_if and A_ff of one layer in 64 bits."""
    shape = frames, text, n_vis, cu = _shape(case)
    q, k, v = _inputs(case, seed, layer)
    hq, hkv, d, npf, tile = case["hq"], case["hkv"], case["d"], case["npf"], case["tile"]
    gq, n = hq // hkv, int(cu[-1])
    f64 = dict(dtype=torch.float64, device="cuda")
    o, lse = torch.zeros((n, hq, d), **f64), torch.zeros((hq, n), **f64)
    tok = torch.zeros((hq, int(n_vis.sum())), **f64)
    cues = case["kind"] == "cues"
    aif, aff = [], []
    r = 0
    for b in range(len(frames)):
        s, nv, t, T = int(cu[b]), int(n_vis[b]), text[b], frames[b]
        keep = _sets(q, k, case, b, shape)[0] if case["kind"] == "sparse" else None
        vis0 = int(n_vis[:b].sum())
        a_if, a_ff = torch.zeros((T, npf, npf), **f64), torch.zeros((T, T), **f64)
        kd = [k[s:s + nv + t, g].double() for g in range(hkv)]
        vd = [v[s:s + nv + t, g].double() for g in range(hkv)]
        for a in list(range(0, nv, tile)) + [nv + x for x in range(0, t, tile)]:
            e = min(a + tile, nv if a < nv else nv + t)
            if a >= nv or case["kind"] == "sparse":
                cols = torch.arange(e, device="cuda")
            else:
                cols = torch.cat([torch.arange(c * tile, min((c + 1) * tile, nv), device="cuda")
                                  for c in mask[1][mask[0][r]:mask[0][r + 1]]])
            r += a < nv
            rows = torch.arange(a, e, device="cuda")
            ok = (cols[None] <= rows[:, None])[None].expand(gq, -1, -1)
            blk = torch.where(cols < nv, cols // case["block"], nv // case["block"] + (cols - nv) // case["block"])
            for g in range(hkv):
                sc = (q[s + a:s + e, g * gq:(g + 1) * gq].double().transpose(0, 1) @ kd[g][cols].T) / math.sqrt(d)
                allowed = ok if keep is None else ok & keep[g * gq:(g + 1) * gq, a:e][:, :, blk]
                sc = sc.masked_fill(~allowed, -math.inf)
                ls = torch.logsumexp(sc, 2)
                p = torch.exp(sc - ls[..., None])
                o[s + a:s + e, g * gq:(g + 1) * gq] = (p @ vd[g][cols]).transpose(0, 1)
                lse[g * gq:(g + 1) * gq, s + a:s + e] = ls
                if a >= nv:
                    tok[g * gq:(g + 1) * gq, vis0:vis0 + nv] += p[:, :, :nv].sum(1)
                elif cues:
                    m = p.sum(0)
                    by_row = m.view((e - a) // npf, npf, len(cols)).sum(1)
                    to = torch.div(cols, npf, rounding_mode="floor")
                    a_ff[a // npf:e // npf].index_add_(1, to, by_row)
                    at = {int(c): i for i, c in enumerate(cols[::npf].tolist())}
                    for fr in range(a // npf, e // npf):
                        i = at[fr * npf] * npf
                        a_if[fr] += m[fr * npf - a:(fr + 1) * npf - a, i:i + npf]
        aif.append(a_if / hq)
        aff.append(torch.tril(a_ff, -1)[1:, :-1] / (npf * hq) if T > 1 else torch.zeros((0, 0), **f64))
    return o, lse, tok, torch.cat(aif), aff


def _exact_maps(case, tok):
    frames, text, n_vis, _ = _shape(case)
    frame = tok.view(case["hq"], sum(frames), case["npf"]).sum(2)
    head, aqf, f0 = [], [], 0
    for f, t in zip(frames, text):
        part = frame[:, f0:f0 + f]
        head.append(part.sum(1))
        aqf.append(part.sum(0) / (case["hq"] * t))
        f0 += f
    return [tok, frame, torch.stack(head), torch.cat(aqf)]


def _exact_coarse(case, seed):
    shape = frames, text, n_vis, cu = _shape(case)
    q, k, _ = _inputs(case, seed)
    hq, hkv, d, B = case["hq"], case["hkv"], case["d"], case["block"]
    toks = []
    for b in range(len(frames)):
        s, nv, t = int(cu[b]), int(n_vis[b]), text[b]
        keep, kbar, own = _sets(q, k, case, b, shape)
        nvb, pos = nv // B, torch.arange(nv, nv + t, device="cuda")
        cols = torch.arange(nv + t, device="cuda")
        blk = torch.where(cols < nv, cols // B, nvb + (cols - nv) // B)
        tok = torch.empty((hq, nv), dtype=torch.float64, device="cuda")
        for h in range(hq):
            g = h // (hq // hkv)
            qt = q[s + nv:s + nv + t, h].double()
            coarse = ((qt @ kbar[:, g].T) / math.sqrt(d))[:, blk]
            exact_ = (qt @ k[s:s + nv + t, g].double().T) / math.sqrt(d)
            mine = own[pos][:, None] == blk[None]
            a = torch.where(mine, exact_, coarse)
            ok = keep[h, pos][:, blk] & (~mine | (cols[None] <= pos[:, None]))
            tok[h] = torch.softmax(a.masked_fill(~ok, -math.inf), 1)[:, :nv].sum(0)
        toks.append(tok)
    return {"maps": _exact_maps(case, torch.cat(toks, 1))}


def exact(case, seed):
    if case["kind"] == "retain":
        return None                      # whole numbers: the retained sets themselves
    if case["kind"] == "coarse":
        return _exact_coarse(case, seed)
    mask = None if case["kind"] == "sparse" else _mask(case, seed)
    layers, tok, aif, aff = [], 0.0, None, None
    for i in range(case["layers"]):
        o, lse, t, aif, aff = _exact_layer(case, seed, i, mask)
        layers.append((o, lse))
        tok = tok + t
    out = {"layers": layers, "maps": _exact_maps(case, tok)}
    if case["kind"] == "cues":
        eff = []
        for f, x in zip(_shape(case)[0], aff):
            e = torch.zeros((f,), dtype=torch.float64, device="cuda")
            if f > 1:
                e[1:] += x.sum(1)
                e[:-1] += x.sum(0)
            eff.append(0.5 * e)
        out.update(aif=aif, aff=torch.cat([x.reshape(-1) for x in aff]), eff=torch.cat(eff))
    return out
