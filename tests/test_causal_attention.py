"""The causal tcgen05 attention kernel of training-time test against the CPU oracle, at the edges of its tiles."""
import numpy as np
import pytest
import torch

import parity
import pyoracle as po
from paper_2503_01840_b200 import binding as sb
from paper_2503_01840_b200 import synth

pytestmark = pytest.mark.gpu

@pytest.mark.parametrize("T,H,G,J,ps,shift", [(1, 8, 2, 2, 16, 0), (127, 2, 2, 1, 32, 0), (256, 6, 2, 0, 64, 0), (257, 4, 4, 3, 16, 0),
                                              (385, 3, 1, 2, 16, 0), (384, 8, 2, 3, 64, 0), (200, 4, 2, 3, 16, 4), (130, 3, 3, 8, 32, 4),
                                              (100, 4, 4, 7, 16, 0), (320, 2, 2, 8, 32, 0), (700, 1, 1, 5, 64, 0), (200, 4, 1, 5, 16, 0), (129, 4, 2, 1, 16, 0)])
def test_causal_kernel_edges_vs_oracle(T, H, G, J, ps, shift):
    """One position, whole and ragged tiles, both ways of pairing query tiles, the three page sizes, and diagonal entries
    that start on an 8-byte boundary only (shift elements into their allocation)."""
    hd = 128
    g = torch.Generator().manual_seed(T * 7 + J)

    def rand(*s):
        return torch.randn(*s, generator=g).to(torch.bfloat16)

    q, k0, v0 = rand(T, H, hd), rand(T, G, hd), rand(T, G, hd)
    kd, vd = (rand(J, T, G, hd), rand(J, T, G, hd)) if J else (None, None)
    pages = (T + ps - 1) // ps
    perm = torch.randperm(pages + 2, generator=g)[:pages].to(torch.int32)
    kp, vp = torch.zeros(pages + 2, G, ps, hd, dtype=torch.bfloat16), torch.zeros(pages + 2, G, ps, hd, dtype=torch.bfloat16)
    for p_ in range(T):
        kp[perm[p_ // ps], :, p_ % ps] = k0[p_]
        vp[perm[p_ // ps], :, p_ % ps] = v0[p_]

    def dev(t):
        buf = torch.empty(t.numel() + shift, dtype=torch.bfloat16, device="cuda")
        buf[shift:] = t.flatten().cuda()
        return buf[shift:].view(t.shape)

    out, lse = sb.ttt_attention(q.cuda(), kp.cuda(), vp.cuda(), perm.cuda(), dev(kd) if J else None, dev(vd) if J else None, want_lse=True)
    zero = np.zeros((0, T, G, hd))
    o_out, o_lse = po.ttt_attention_rows(q.float().numpy(), k0.float().numpy(), v0.float().numpy(), kd.float().numpy() if J else zero,
                                         vd.float().numpy() if J else zero, list(range(T)))
    # outputs of order 1: bf16 output and bf16 probabilities, 2^-9 each; the statistics are fp32
    assert np.abs(out.float().cpu().numpy() - o_out).max() < 2e-2
    assert np.abs(lse.cpu().numpy() - o_lse).max() < 1e-4


@pytest.mark.parametrize("T,H,G", [(130, 4, 1), (200, 2, 2)])
def test_rows_whose_scores_are_all_minus_infinity(T, H, G):
    """An infinite query component against keys that are all negative there: the row's output is 0 and its normaliser -inf;
    the other rows are what they are without it."""
    g = torch.Generator().manual_seed(T)
    q, k, v = (torch.randn(*s, generator=g).to(torch.bfloat16).cuda() for s in ((T, H, 128), (-(-T // 16), G, 16, 128), (-(-T // 16), G, 16, 128)))
    k[..., 5] = -1.0 - k[..., 5].abs()
    table = torch.arange(k.shape[0], dtype=torch.int32, device="cuda")
    out, lse = sb.ttt_attention(q, k, v, table, None, None, want_lse=True)
    bad = torch.zeros(T, H, dtype=torch.bool, device="cuda")
    for r, h in ((0, 0), (70, 1), (T - 1, H - 1)):
        q[r, h, 5], bad[r, h] = float("inf"), True
    out2, lse2 = sb.ttt_attention(q, k, v, table, None, None, want_lse=True)
    assert (out2[bad] == 0).all() and (lse2[bad] == -float("inf")).all()
    assert torch.equal(out2[~bad], out[~bad]) and torch.equal(lse2[~bad], lse[~bad]) and torch.isfinite(lse).all()


@pytest.mark.parametrize("T,H,G,J", [(40, 2, 1, 0), (128, 4, 1, 2), (300, 2, 2, 1), (513, 4, 4, 0)])
def test_softmax_warps_that_come_late(T, H, G, J):
    """Warps that look for a tile's last contraction long after it completed (one to nine key steps per tile) find it
    complete, and the outputs are the same bits."""
    g = torch.Generator().manual_seed(T)
    pages = -(-T // 16)
    q, k, v = (torch.randn(*s, generator=g).to(torch.bfloat16).cuda() for s in ((T, H, 128), (pages, G, 16, 128), (pages, G, 16, 128)))
    kd, vd = (torch.randn(J, T, G, 128, generator=g).to(torch.bfloat16).cuda() for _ in range(2)) if J else (None, None)
    table = torch.arange(pages, dtype=torch.int32, device="cuda")
    run = lambda: sb.ttt_attention(q, k, v, table, kd, vd, want_lse=True)
    out, lse = run()
    sb.lib().spec_debug_causal(1)
    try:
        late, late_lse = run()
        torch.cuda.synchronize()
    finally:
        sb.lib().spec_debug_causal(0)
    assert torch.isfinite(lse).all() and torch.equal(out, late) and torch.equal(lse, late_lse)


@pytest.mark.parametrize("T,H,G,J", [(130, 4, 1, 0), (300, 8, 2, 3), (513, 4, 4, 2)])
def test_training_time_test_wait_that_runs_out_gives_nan(T, H, G, J):
    """The first CTA never receives its queries (test hook): its rows, those of the last positions of its heads, are NaN, all
    others are untouched, and the next call is whole."""
    g = torch.Generator().manual_seed(T)
    pages = -(-T // 16)
    q, k, v = (torch.randn(*s, generator=g).to(torch.bfloat16).cuda() for s in ((T, H, 128), (pages, G, 16, 128), (pages, G, 16, 128)))
    kd, vd = (torch.randn(J, T, G, 128, generator=g).to(torch.bfloat16).cuda() for _ in range(2)) if J else (None, None)
    table = torch.arange(pages, dtype=torch.int32, device="cuda")
    run = lambda: sb.ttt_attention(q, k, v, table, kd, vd, want_lse=True)
    out, lse = run()
    sb.lib().spec_debug_causal(2)
    try:
        lost, lost_lse = run()
        torch.cuda.synchronize()
    finally:
        sb.lib().spec_debug_causal(0)
    block, heads = (128, 2) if (H // G) % 2 == 0 else (256, 1)
    gone = torch.zeros(T, H, dtype=torch.bool, device="cuda")
    gone[(T - 1) // block * block :, :heads] = True
    assert torch.isnan(lost[gone]).all() and torch.isnan(lost_lse[gone]).all()
    assert torch.equal(lost[~gone], out[~gone]) and torch.equal(lost_lse[~gone], lse[~gone])
    again, again_lse = run()
    assert torch.equal(again, out) and torch.equal(again_lse, lse)


def test_prefill_wait_that_runs_out_is_reported():
    """The same in a prefill: it returns SPEC_ERR_DEVICE_STATUS with the site of the wait, and the next one is whole."""
    cfg = synth.ModelCfg("wait", "bf16", 2, 512, 8, 2, 128, 1408, 2048, 1024, (0, 0, 1), 5e5, batch=2, tree_depth=2, tree_topk=4, tree_nodes=12, seed=9)
    tw, dw = parity.to_dev(synth.make_target_weights(cfg)), parity.to_dev(synth.make_draft_weights(cfg))
    rng = np.random.default_rng(1)
    prompts = [rng.integers(0, cfg.vocab, n).astype(np.int32) for n in (300, 77)]
    dec = sb.SpecDecoder(cfg, tw, dw, batch=2, max_ctx=400)
    first = dec.prefill(prompts, 8)
    steps = dec.step()
    sb.lib().spec_debug_causal(2)
    try:
        with pytest.raises(sb.SpecError) as e:
            dec.prefill(prompts, 8)
    finally:
        sb.lib().spec_debug_causal(0)
    assert e.value.code == -7 and "site 43" in str(e.value), str(e.value)
    assert np.array_equal(dec.prefill(prompts, 8), first) and all(np.array_equal(a, b) for a, b in zip(dec.step(), steps))
    dec.close()


@pytest.mark.parametrize("T,H,bound", [(256, 16, 1.93e-3), (512, 16, 2.06e-3), (1500, 8, 2.045e-3)])
def test_error_against_fp64(T, H, bound):
    """Relative error (2-norm) over all outputs.  Rounding the output to bf16 makes 1.66e-3 of it, rounding the probabilities
    the rest; with a reference maximum that follows the row's only by jumps of 2^8 it is 1.96e-3, 2.08e-3 and
    2.06e-3."""
    g = torch.Generator().manual_seed(T)
    pages = -(-T // 16)
    q, k, v = (torch.randn(*s, generator=g).to(torch.bfloat16).cuda() for s in ((T, H, 128), (pages, H, 16, 128), (pages, H, 16, 128)))
    out = sb.ttt_attention(q, k, v, torch.arange(pages, dtype=torch.int32, device="cuda"), None, None).double()
    K, V = (t.double().permute(1, 0, 2, 3).reshape(H, pages * 16, 128)[:, :T] for t in (k, v))
    s = torch.einsum("thd,hkd->htk", q.double(), K) / 128 ** 0.5
    s.masked_fill_(torch.ones(T, T, dtype=torch.bool, device="cuda").triu(1), -float("inf"))
    ref = torch.einsum("htk,hkd->thd", s.softmax(-1), V)
    rel = ((out - ref).norm() / ref.norm()).item()
    assert rel < bound, rel


@pytest.mark.parametrize("T,H,G", [(65, 2, 2), (400, 4, 1), (900, 2, 1), (901, 3, 3)])
def test_maxima_that_rise_with_the_keys(T, H, G):
    """Rows whose maximum rises by more than 2^8 every three 64-key steps, to the last of them, beside rows (every other one) whose
    scores stay small: the first rescale their sums again and again, the second are what they are without them."""
    g = torch.Generator().manual_seed(T)
    pages = -(-T // 16)
    q, k, v = (torch.randn(*s, generator=g).to(torch.bfloat16).cuda() for s in ((T, H, 128), (pages, G, 16, 128), (pages, G, 16, 128)))
    q[::2, :, 3], q[1::2, :, 3] = 8.0, 0.0
    k[..., 3] = ((torch.arange(pages * 16, device="cuda") // 64) * 4).view(pages, 1, 16).to(torch.bfloat16)      # exact: 0, 4, 8, ...
    out, lse = sb.ttt_attention(q, k, v, torch.arange(pages, dtype=torch.int32, device="cuda"), None, None, want_lse=True)
    K, V = (t.double().permute(1, 0, 2, 3).reshape(G, pages * 16, 128)[:, :T].repeat_interleave(H // G, 0) for t in (k, v))
    s = torch.einsum("thd,hkd->htk", q.double(), K) / 128 ** 0.5
    s.masked_fill_(torch.ones(T, T, dtype=torch.bool, device="cuda").triu(1), -float("inf"))
    # outputs of order 1: bf16 output and bf16 probabilities, 2^-9 each; scores to 50, sums of fp32 terms: 50 * 2^-24 and 2^-22 an exponential
    assert (out.double() - torch.einsum("htk,hkd->thd", s.softmax(-1), V)).abs().max() < 2e-2
    assert (lse.double() - torch.logsumexp(s, -1).T).abs().max() < 1e-4
