"""GPU parity of the text rows' evidence sums formed by evisel_evidence_reduce
(evisel_probe_args.text_evidence = 1): the token / frame / head maps and A_qf
from q, k and the probe's LSE against the float64 oracle on the seeded
workloads and edge cases, summed over layers, and through the entry point that
allocates nothing (the 65K probe fits its 64 MiB scratch in this mode); and
both modes (in the probe call, in the evidence call: one kernel) against sums
in float64 from the same q, k and LSE.

Tolerances: the oracle's (frame evidence <= 1e-3 abs per entry, identical top-k
planted frames). With the LSE given, what is left is the rounding of s and LSE
in log2 units (|s| < 2^5: below 2^-18 absolute, so 4e-6 relative in the
exponential), the exponential's own 2^-22 and at most 256 fp32 additions
(256 * 2^-24): 2e-5 of the largest entry.
"""
import numpy as np
import pytest

import oracle
from paper_2608_05780_gb300 import _binding as B
from paper_2608_05780_gb300 import workloads as wl
from gpu_helpers import check_maps, np32, oracle_maps, run_cuda, to_device

pytestmark = pytest.mark.gpu


def _maps(out):
    return [np32(out[k]) for k in ("tok", "frame", "head", "aqf")]


@pytest.mark.parametrize("name", ["tiny", "single", "long65k", "varlen8"])
def test_recompute_maps_match_oracle(cuda_lib, name):
    probe = wl.make_probe(wl.CONFIGS[name])
    out, ws = run_cuda(cuda_lib, probe, text_evidence=True)
    ws.free()
    check_maps(_maps(out), oracle_maps(probe), probe, label=f"{name} recompute")


def _sums_float64(probe, lse):
    """The four maps in float64 from bf16 q and k and the given LSE, in torch."""
    import torch
    cfg = probe.cfg
    q, k, _ = to_device(probe)
    npf, gq = cfg.tokens_per_frame, cfg.hq // cfg.hkv
    tok = []
    for b, nv in enumerate(int(x) for x in probe.n_vis):
        a, e = int(probe.cu_seqlens[b]), int(probe.cu_seqlens[b + 1])
        heads = []
        for h in range(cfg.hq):
            s = q[a + nv:e, h].double() @ k[a:a + nv, h // gq].double().T * q.shape[2] ** -0.5
            heads.append((s - lse[h, a + nv:e, None].double()).exp().sum(0))
        tok.append(torch.stack(heads))
    frame = [t.reshape(cfg.hq, -1, npf).sum(2) for t in tok]
    text = np.diff(probe.cu_seqlens) - probe.n_vis
    return dict(tok=torch.cat(tok, 1), frame=torch.cat(frame, 1), head=torch.stack([f.sum(1) for f in frame]),
                aqf=torch.cat([f.sum(0) / (cfg.hq * int(t)) for f, t in zip(frame, text)]))


@pytest.mark.parametrize("name", ["single", "long65k", "varlen8"])
def test_both_modes_match_float64_sums(cuda_lib, name):
    probe = wl.make_probe(wl.CONFIGS[name])
    a, ws = run_cuda(cuda_lib, probe)
    ws.free()
    b, ws = run_cuda(cuda_lib, probe, text_evidence=True)
    ws.free()
    for k in ("o", "lse"):
        assert np.array_equal(np32(a[k]), np32(b[k])), k      # the attention itself is unchanged
    want = _sums_float64(probe, a["lse"])
    for k in ("tok", "frame", "head", "aqf"):
        scale = max(want[k].abs().max().item(), 1e-30)
        for out in (a, b):
            err = (out[k].double() - want[k]).abs().max().item()
            assert err <= 2e-5 * scale, (k, err, scale)


EDGE = {
    "ragged_tiles_t128_d128": dict(frames=(44,), n_text=(77,), hq=8, hkv=2, d=128, tile=128, window=3),
    "t64_d64_long_text": dict(frames=(36,), n_text=(300,), hq=4, hkv=1, d=64, tile=64, window=2),
    "odd_group_t64": dict(frames=(20,), n_text=(40,), hq=6, hkv=2, d=64, tile=64, window=2),
    "npf64_t128": dict(frames=(9,), n_text=(40,), npf=64, hq=4, hkv=2, d=128, tile=128, window=2),
    "npf4": dict(frames=(70,), n_text=(20,), npf=4, hq=4, hkv=2, d=64, tile=64, window=2),
    "varlen_mixed": dict(frames=(3, 0, 17, 8), n_text=(12, 40, 0, 130), hq=4, hkv=2, d=128, tile=128, window=2),
    "sharp": dict(frames=(40,), n_text=(60,), hq=4, hkv=2, d=128, tile=128, window=4, sharp=True),
}


@pytest.mark.parametrize("name", sorted(EDGE))
def test_recompute_edge_cases(cuda_lib, name):
    from test_gpu_parity import _custom
    probe = _custom(**EDGE[name])
    out, ws = run_cuda(cuda_lib, probe, text_evidence=True)
    ws.free()
    check_maps(_maps(out), oracle_maps(probe), probe, label=f"{name} recompute")


def test_recompute_accumulates_over_layers(cuda_lib):
    cfg = wl.CONFIGS["depth28"]
    mask = wl.build_mask(cfg)
    ws = maps = ref = None
    for layer in range(3):
        probe = wl.make_probe(cfg, layer, mask=mask)
        out, ws = run_cuda(cuda_lib, probe, ws=ws, maps=maps, accumulate=layer > 0, text_evidence=True)
        maps = [out[k] for k in ("tok", "frame", "head", "aqf")]
        r = oracle_maps(probe)
        ref = r if ref is None else [a + b for a, b in zip(ref, r)]
    check_maps([np32(m) for m in maps], ref, probe, label="3 layers recompute")
    ws.free()


def test_noalloc_recompute_fits_the_65k_probe(cuda_lib):
    """In this mode the 65,664-token probe fits the no-alloc scratch."""
    import torch
    probe = wl.make_probe(wl.CONFIGS["long65k"])
    cfg = probe.cfg
    ref, ws = run_cuda(cuda_lib, probe)
    ws.free()
    q, k, v = to_device(probe)
    n, hq, d = q.shape
    total_vis = int(np.sum(probe.n_vis))
    frames = total_vis // cfg.tokens_per_frame
    o = torch.empty((n, hq, d), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((hq, n), device="cuda")
    tok = torch.full((hq, total_vis), float("nan"), device="cuda")
    frame = torch.full((hq, frames), float("nan"), device="cuda")
    head = torch.full((1, hq), float("nan"), device="cuda")
    aqf = torch.full((frames,), float("nan"), device="cuda")
    status = B.evisel_probe_evidence_noalloc(q, k, v, probe.cu_seqlens, probe.n_vis, cfg.tokens_per_frame, cfg.tile,
                                             probe.row_ptr, probe.col_idx, o, lse, tok, frame, head, aqf,
                                             text_evidence=True)
    assert status == 0
    assert np.array_equal(o.float().cpu().numpy(), np32(ref["o"]))
    for got, want in ((tok, ref["tok"]), (frame, ref["frame"]), (head, ref["head"]), (aqf, ref["aqf"])):
        x, y = np32(got).astype(np.float64), np32(want).astype(np.float64)
        assert np.all(np.isfinite(x))
        assert np.abs(x - y).max() <= 2e-5 * max(np.abs(y).max(), 1e-30)
