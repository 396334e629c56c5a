"""Kernel variants and dispatch branches at the sizes where each can go wrong: edges of tiles, MMA
widths, pieces and batches, the smallest and largest of a range.  Against the float64 oracle under
the tolerances of ``tests.parity``; paged caches against the dense call, bit for bit.
"""
import numpy as np
import pytest
import torch

import paper_2608_13076_gb300 as spade
from paper_2608_13076_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev(gpu_lib):
    return torch.device("cuda:0")


def _spec(name, seed, **over):
    base = dict(B=1, Hq=4, Hkv=2, D=128, H=256, V=1000, ctx=(1, 90), k=(0, 0), mode="greedy", seed=seed)
    return W.WorkloadSpec(name, **{**base, **over})


# The projection.  At most 128 rows: a cluster of two CTAs per range of rotary pairs, each with half
# of the k-chunks (H = 64: one of them has none).  More rows over wide layers (at least eight quads
# of pairs per cluster): a second MMA chunk above 256 rows, the exchange in two to four batches.
# More rows over narrow layers, or more than fit the ring (464 rows are the most that do, with 8 quads per
# cluster): the form with partial sums in a workspace.
QKV = {
    "one_row_one_chunk": dict(H=64),
    "n16": dict(B=2, k=(7, 7), H=72),
    "n17_d64": dict(B=1, k=(16, 16), H=136, D=64, Hq=6),
    "rows128": dict(B=16, k=(7, 7), H=520, Hq=32, Hkv=4),
    "rows129_wide": dict(B=3, k=(42, 42), H=200, Hq=32, Hkv=4),
    "rows256_wide": dict(B=32, k=(7, 7), H=128, Hq=32, Hkv=8),
    "rows272_wide_d64": dict(B=34, k=(7, 7), H=192, D=64, Hq=60, Hkv=10),
    "rows389_wide": dict(B=64, k=(1, 10), H=200, Hq=40, Hkv=8),
    "rows464_wide": dict(B=58, k=(7, 7), H=128, Hq=28, Hkv=4),
    "rows512_past_the_ring": dict(B=64, k=(7, 7), H=128, Hq=32, Hkv=4),
    # four batches, the last of one row: CTA 1 of each cluster receives nothing of it
    "rows193_four_batches": dict(B=1, k=(192, 192), H=128, Hq=58, Hkv=29),
    "rows193_four_batches_d64": dict(B=193, H=128, D=64, Hq=216, Hkv=8),
    "rows129_narrow": dict(B=3, k=(42, 42), H=200),
}


@pytest.mark.parametrize("name", sorted(QKV))
def test_qkv_forms(dev, name):
    spec = _spec(name, 300 + len(name), **QKV[name])
    wl = W.make_workload(spec, device=dev, cache_pad=3)
    x, w = W.make_qkv_inputs(spec, wl["R"], device=dev)
    pg = W.to_paged(wl, 64, seed=5)
    k0, v0 = wl["k_cache"].clone(), wl["v_cache"].clone()
    q, st = parity.gpu_qkv_rope(wl, x, w)
    qp, stp = torch.full_like(q, float("nan")), spade.status_tensor(dev)
    ws = spade.qkv_workspace(wl["R"], wl["Hq"], wl["Hkv"], wl["D"], device=dev)
    spade.spade_verify_qkv_rope_paged(x, w, pg["block_table"], wl["ctx_lens"], wl["n_draft"], wl["cu_q"], qp,
                                      pg["k_pool"], pg["v_pool"], Hq=wl["Hq"], rope_theta=spec.rope_theta,
                                      max_k=int(wl["n_draft"].max()), workspace=ws, status=stp)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and int(stp.item()) == 0
    parity.check_qkv_rope(wl, x, w, q, k0, v0)
    assert torch.equal(qp, q)
    for b in range(wl["B"]):  # the verify slots, page by page
        lo, n = int(wl["ctx_lens"][b]), int(wl["n_draft"][b]) + 1
        for s in range(lo, lo + n):
            page = int(pg["block_table"][b, s // 64])
            assert torch.equal(pg["k_pool"][page, :, s % 64], wl["k_cache"][b, :, s])
            assert torch.equal(pg["v_pool"][page, :, s % 64], wl["v_cache"][b, :, s])


# The LM head.  Row counts around the statistics' blocks of 16, around the one-launch limit, and the
# most rows of the two-launch form; slices that end inside a tile and inside a warp's 32 entries.
ROWS = {"r1": (1, 0, 1), "r16": (2, 7, 1), "r17": (1, 16, 1), "r256": (32, 7, 1), "r257": (1, 256, 2),
        "r400": (50, 7, 2), "r512": (64, 7, 2)}


@pytest.mark.parametrize("mode", ["greedy", "stochastic"])
@pytest.mark.parametrize("name", sorted(ROWS))
def test_lm_head_row_counts(dev, name, mode):
    B, k, launches = ROWS[name]
    wl = W.make_workload(_spec(name, 320 + B, B=B, k=(k, k), V=9003, mode=mode, target_accept=0.7), device=dev)
    B, R, H, V = wl["B"], wl["R"], wl["H"], wl["V"]
    assert spade.spade_accept_launches(B, R, H, V) == launches
    ws = spade.accept_workspace(B, R, H, V, device=dev)
    acc, tok, st = parity.gpu_accept(wl, workspace=ws)
    torch.cuda.synchronize()
    assert int(st.item()) & ~spade.DEV_FALLBACK == 0
    logits = parity.oracle_logits(wl)
    cmp = parity.compare_accept(acc, tok, parity.oracle_accept_from_logits(wl, logits))
    assert cmp["mismatch_unflagged"] == 0 and cmp["flagged"] <= B // 8, cmp
    worst = parity.compare_row_stats(spade.read_accept_stats(ws, B, R, H, V), logits, wl)
    assert worst["argmax_mismatch"] == 0 and max(worst["max"], worst["lse"], worst["draft_logit"]) <= 1.0, worst


# The one-launch form takes what 512 accumulator columns hold: tiles per slice x rows (rounded up to 8).
# (sizes, most rows in one launch) for the 152 slices of a GB300
@pytest.mark.parametrize("V,most", [(19456, 256), (32000, 256), (64000, 128), (128256, 72), (152064, 64)])
def test_lm_head_form(dev, V, most):
    if torch.cuda.get_device_properties(dev).multi_processor_count != 152:
        pytest.skip("limits computed for 152 slices")
    assert [spade.spade_accept_launches(1, r, 256, V) for r in (most, most + 1)] == [1, 2]


# A slice that the pair kernel sums with its partner is summed in the order of the one-launch form
# with stages of two chunks (up to 80 rows): same bits.  Here 8 of 152 slices have no partner.
def test_pairs_sum_as_one_launch(dev):
    wl = W.make_workload(_spec("order", 330, B=65, k=(3, 3), H=1280, V=20000), device=dev)
    n, B = 64, 16
    part = dict(wl, B=B, R=n, hidden=wl["hidden"][:n].contiguous(), draft_tokens=wl["draft_tokens"][:n - B].contiguous(),
                uniforms=wl["uniforms"][:n].contiguous(), mode=wl["mode"][:B].contiguous(),
                cu_q=wl["cu_q"][:B + 1].contiguous(), n_draft=wl["n_draft"][:B].contiguous())
    maxima = []
    for w, launches in ((wl, 2), (part, 1)):
        assert spade.spade_accept_launches(w["B"], w["R"], w["H"], w["V"]) == launches
        ws = spade.accept_workspace(w["B"], w["R"], w["H"], w["V"], device=dev)
        parity.gpu_accept(w, workspace=ws)
        torch.cuda.synchronize()
        maxima.append(spade.read_accept_stats(ws, w["B"], w["R"], w["H"], w["V"])["max"][:n])
    assert float((maxima[0] == maxima[1]).float().mean()) > 0.8


# The draw.  Shares of one piece and of several (more than 8192 entries: two buffers, and the owner's
# piece again), groups of one CTA and of more, q rows that bulk copies can and cannot read.
DRAW = {
    "one_cta_one_piece": dict(B=2, k=(4, 4), V=1024),
    "one_cta_three_pieces": dict(B=80, k=(1, 1), V=20000),
    "one_cta_unaligned": dict(B=80, k=(1, 1), V=20001),
    "two_ctas_unaligned": dict(B=60, k=(2, 2), V=33002),
    "two_launches_aligned": dict(B=60, k=(4, 4), V=40000),
    "two_launches_unaligned": dict(B=60, k=(4, 4), V=40003),
    "two_launches_one_cta": dict(B=130, k=(1, 2), V=20004),
}


@pytest.mark.parametrize("name", sorted(DRAW))
def test_draw_shares(dev, name):
    spec = _spec(name, 340 + len(name), H=128, mode="stochastic", target_accept=0.7, logit_scale=4.0, **DRAW[name])
    wl = W.make_workload(spec, device=dev)
    if name.startswith("two_launches"):
        assert spade.spade_accept_launches(wl["B"], wl["R"], wl["H"], wl["V"]) == 2
    acc, tok, st = parity.gpu_accept(wl)
    torch.cuda.synchronize()
    assert int(st.item()) & ~spade.DEV_FALLBACK == 0
    cmp = parity.compare_accept(acc, tok, parity.oracle_accept(wl))
    assert cmp["mismatch_unflagged"] == 0 and cmp["flagged"] < wl["B"] // 2, cmp


# A target before the last piece of a share: its piece is copied and turned into terms once more, and
# the walk reads the terms that other lanes of the warp have just stored.
@pytest.mark.parametrize("B,k,V", [(80, 1, 20000), (80, 1, 20001), (130, 1, 20004)])
def test_draw_piece_again(dev, B, k, V):
    spec = _spec("again", 355 + V % 7, B=B, k=(k, k), V=V, H=128, mode="stochastic", target_accept=0.7, logit_scale=2.0)
    wl = W.make_workload(spec, device=dev)
    wl["uniforms"][wl["cu_q"][1:].long() - 1] = torch.linspace(0.01, 0.75, B, device=dev)
    ref = parity.oracle_accept(wl)
    assert int((ref["next_token"] < 2 * 8192).sum()) > B // 2
    ws = spade.accept_workspace(B, wl["R"], wl["H"], V, device=dev)
    for _ in range(8):
        acc, tok, st = parity.gpu_accept(wl, workspace=ws)
        torch.cuda.synchronize()
        assert int(st.item()) & ~spade.DEV_FALLBACK == 0
        cmp = parity.compare_accept(acc, tok, ref)
        assert cmp["mismatch_unflagged"] == 0 and cmp["flagged"] < B // 2, cmp


# Every row of a call leaves its statistics, also rows past the last sequence's (padding of a captured
# call) and of a sequence that is reported: what an earlier call left there must not stay.
@pytest.mark.parametrize("B,k,V", [(6, 4, 1000), (6, 4, 5000), (60, 4, 5000)])
def test_statistics_of_every_row(dev, B, k, V):
    wl = W.make_workload(_spec("rest", 370 + B, B=B, k=(k, k), V=V, mode="mixed", target_accept=0.7), device=dev)
    R, H = wl["R"], wl["H"]
    assert spade.spade_accept_launches(B, R, H, V) == (2 if B == 60 else 1)
    ws = spade.accept_workspace(B, R, H, V, device=dev)
    other = dict(wl, hidden=wl["hidden"].flip(0).contiguous())
    parity.gpu_accept(other, workspace=ws)  # (leaves its own statistics)
    cut, nd = wl["cu_q"].clone(), wl["n_draft"].clone()
    cut[-1] -= 2  # the last sequence is two drafts shorter: two rows of padding
    nd[-1] -= 2
    nd[1] += 1    # reported: its rows and drafts do not agree
    call = dict(wl, cu_q=cut, n_draft=nd)
    acc, tok, st = parity.gpu_accept(call, workspace=ws)
    torch.cuda.synchronize()
    assert int(st.item()) & ~spade.DEV_FALLBACK == spade.DEV_BAD_INDEX
    assert int(acc[1]) == 0 and int(tok[1]) == -1
    logits = parity.oracle_logits(wl)
    stats = spade.read_accept_stats(ws, B, R, H, V)
    worst = parity.compare_row_stats(stats, logits, dict(wl, n_draft=torch.zeros_like(nd)))
    assert worst["argmax_mismatch"] == 0 and max(worst["max"], worst["lse"]) <= 1.0, worst
    assert stats["accept_bit"][(k + 1):2 * (k + 1)].tolist() == [0] * (k + 1) and stats["accept_bit"][-2:].tolist() == [0, 0]


# Vocabularies of at most eight tiles run as one cluster, larger ones as a cooperative grid: one CTA, a
# ragged last tile, the largest cluster and the smallest grid beyond it, with every option at once.
@pytest.mark.parametrize("V", [100, 129, 1024, 1025])
@pytest.mark.parametrize("mode", ["greedy", "mixed"])
def test_small_vocabularies(dev, V, mode):
    spec = _spec("small_v", 350 + V, B=6, k=(0, 5), V=V, mode=mode, target_accept=0.7, logit_scale=3.0)
    wl = W.make_workload(spec, device=dev)
    T, top_p = torch.linspace(0.7, 1.4, 6), torch.linspace(0.5, 1.0, 6)
    before = {k: wl[k].clone() for k in ("k_cache", "v_cache", "ctx_lens", "n_draft")}
    acc, tok, st = parity.gpu_accept_sampling(wl, temperature=T.to(dev), top_p=top_p.to(dev), commit=True)
    torch.cuda.synchronize()
    assert int(st.item()) & ~spade.DEV_FALLBACK == 0
    ref = parity.oracle_accept_from_logits(wl, parity.oracle_logits(wl), temperature=T.numpy(), top_p=top_p.numpy())
    cmp = parity.compare_accept(acc, tok, ref)
    assert cmp["mismatch_unflagged"] == 0 and cmp["flagged"] <= 1, cmp
    parity.check_commit_windows(before, wl["k_cache"], wl["v_cache"], wl["ctx_lens"], acc)


# The nucleus search.  Flat logits put nearly every entry in one bin of the first round, so the kept
# lists overflow and the values are read again; one CTA per group (nothing exchanged) and several.
def _nuclei(l, top_p):
    """What a search that tells logits apart to two key steps (2^-14, wider than the fp32 logits' own error) may
    keep of softmax(l): (p, smallest set, its mass, largest set, its mass), as masks over the vocabulary."""
    p = np.exp(l - l.max())
    p /= p.sum()
    order = np.argsort(-l, kind="stable")
    tau = l[order[np.searchsorted(np.cumsum(p[order]), top_p)]]
    least, most = l >= tau + 2.0 ** -14, l >= tau - 2.0 ** -14
    return p, least, p[least].sum(), most, p[most].sum()


@pytest.mark.parametrize("B,V", [(2, 160000), (80, 20000)])
def test_top_p_flat(dev, B, V):
    """Nuclei of tens of thousands of tokens, whose boundary no margin can fix: every accept test and every drawn
    token must follow from some nucleus between the smallest and the largest that two key steps allow."""
    k = 3 if B == 2 else 1
    wl = W.make_workload(_spec("topp_flat", 360 + B, B=B, k=(k, k), H=128, V=V, mode="stochastic", target_accept=0.6,
                               logit_scale=0.05))
    top_p = np.linspace(0.4, 0.9, B)
    logits, q, u = parity.oracle_logits(wl), parity.to_np(wl["draft_probs"]).astype(np.float64), wl["uniforms"]
    tests, rows = [], []
    for b in range(B):
        for i in range(k + 1):
            r = b * (k + 1) + i
            rows.append(_nuclei(logits[r], top_p[b]))
            p, least, s_least, most, s_most = rows[-1]
            if i == k:
                continue
            d = int(wl["draft_tokens"][r - b])
            lo, hi = least[d] * p[d] / s_most, most[d] * p[d] / s_least  # the accept threshold times q(d)
            # uniforms a tenth away from the threshold (rejections where it is below 0.9)
            x = lo / q[r - b, d]
            u[r] = 0.9 * x if x >= 0.9 or r % 3 else 1.1 * x
            u[r] = min(float(u[r]), 1.0 - 2.0 ** -24) if x > 0 else 0.5
            assert most[d] == least[d] and (float(u[r]) * q[r - b, d] < lo or float(u[r]) * q[r - b, d] >= hi)
            tests.append(float(u[r]) * q[r - b, d] < lo)
    assert 0 < sum(tests) < len(tests)
    gpu = {n: v.to(dev) if isinstance(v, torch.Tensor) else v for n, v in wl.items()}
    acc, tok, st = parity.gpu_accept_sampling(gpu, top_p=torch.from_numpy(top_p).float().to(dev))
    torch.cuda.synchronize()
    assert int(st.item()) & ~spade.DEV_FALLBACK == 0
    for b, (a, x) in enumerate(zip(acc.tolist(), tok.tolist())):
        assert a == (tests[b * k:(b + 1) * k] + [False]).index(False), b
        p, least, s_least, most, s_most = rows[b * (k + 1) + a]
        given = q[b * k + a] if a < k else 0.0
        lo = np.cumsum(np.maximum(0.0, least * p / s_most - given))
        hi = np.cumsum(np.maximum(0.0, most * p / s_least - given))
        at = float(u[b * (k + 1) + k])
        # (1e-5: the fp32 terms' own error; the two bounds differ by less than 1 %, so the interval is narrow)
        assert hi[-1] < 1.01 * lo[-1]
        assert most[x] and hi[x] > (at - 1e-5) * lo[-1] and (lo[x - 1] if x else 0.0) < (at + 1e-5) * hi[-1], (b, x)


@pytest.mark.parametrize("B,V", [(80, 3001)])
def test_top_p_peaked(dev, B, V):
    wl = W.make_workload(_spec("topp_lists", 360 + B, B=B, k=(1, 1), H=128, V=V, mode="stochastic", target_accept=0.6,
                               logit_scale=4.0), device=dev)
    top_p = torch.linspace(0.4, 0.9, B)
    acc, tok, st = parity.gpu_accept_sampling(wl, top_p=top_p.to(dev))
    torch.cuda.synchronize()
    assert int(st.item()) & ~spade.DEV_FALLBACK == 0
    ref = parity.oracle_accept_from_logits(wl, parity.oracle_logits(wl), top_p=top_p.numpy())
    cmp = parity.compare_accept(acc, tok, ref)
    assert cmp["mismatch_unflagged"] == 0 and cmp["flagged"] < B // 2, cmp


# After an expired wait every later wait of the block returns at once: 192 of them, each of which may
# suspend its warp for 1 ms if it does not look at the flag first, within 20 ms (64 ms is a third of that).
def test_waits_after_an_expired_one(dev):
    st = spade.status_tensor(dev)
    spade.spade_selftest_wait_timeout(st, 1000)
    torch.cuda.synchronize()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    spade.spade_selftest_wait_timeout(st, 1000)
    t1.record()
    torch.cuda.synchronize()
    assert int(st.item()) == spade.DEV_TIMEOUT
    assert 1.0 <= t0.elapsed_time(t1) < 20.0


# Attention units split into many parts: the merge's batches of four parts and its rows' remainders.
@pytest.mark.parametrize("D,G,k,ctx", [(128, 1, 0, 20000), (64, 1, 0, 700), (128, 5, 6, 9000), (64, 8, 7, 20000),
                                       (128, 8, 7, 600), (128, 3, 8, 330)])
def test_attention_merge(dev, D, G, k, ctx):
    wl = W.make_workload(_spec("merge", 380 + G, Hq=G, Hkv=1, D=D, ctx=(ctx, ctx), k=(k, k)), device=dev)
    out, lse, st = parity.gpu_attention(wl)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    ref, ref_lse = parity.oracle_attention(wl)
    n, bad, worst = parity.compare_attention(out, ref)
    assert bad == 0, worst
    # fp32 sums of at most 20008 exponentials, scores of bf16 products: far below 1e-3
    assert abs(parity.to_np(lse) - ref_lse).max() < 1e-3
