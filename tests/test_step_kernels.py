"""The stochastic acceptance, the launch between two draft passes and the pruning on planted inputs, against the oracle or the rule written out."""
import numpy as np
import pytest
import torch

import pyoracle as po
import step_kernels as sk

pytestmark = pytest.mark.gpu


def _accept(z, u, tok, parent, nn, D, T):
    """z [B][N][V], u [B][2 N], tok / parent [B][N] -> lists of paths and ids."""
    B, N, V = z.shape
    dev = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt).cuda()
    P = D + 1
    out = torch.full((3 * B * P + B,), -7, dtype=torch.int32, device="cuda")
    state = torch.ones(5, B, dtype=torch.int32, device="cuda")
    uu = torch.cat([dev(u, torch.float32).view(-1), torch.tensor([1.0 / T], device="cuda", dtype=torch.float32)])
    mass = torch.zeros(B * N * sk.library().mass_chunks(V), 2, device="cuda")
    rc = sk.call("accept_sampled", dev(z, torch.float32), V, uu, mass, dev(tok, torch.int32), dev(parent, torch.int32), dev(nn, torch.int32), state, out, B, N, D)
    assert rc > 0, rc
    o = out.cpu().numpy()
    path, ids = o[: B * P].reshape(B, P), o[B * P: 2 * B * P].reshape(B, P)
    cnt = o[3 * B * P:]
    assert np.array_equal(state.cpu().numpy()[0], 1 + cnt)
    return [(path[b, : cnt[b]], ids[b, : cnt[b]]) for b in range(B)]


# rejected siblings hold all but `rest` of the root's mass, in one run of 8192 ids or in several
@pytest.mark.parametrize("V,live,rejected", [
    (1000, range(0, 1000), (3, 400, 401)),
    (8192, range(100, 8192), (100, 101, 8191)),
    (20001, range(9000, 20001), (5, 6, 7)),                        # the run that holds the rejected ids has no other
    (20001, range(0, 20001), (5, 8192, 19999)),
    (20000, (4, 9000, 19990), (5, 6, 9001)),
])
@pytest.mark.parametrize("rest", [1e-2, 1e-5, 2e-6])
def test_draw_from_what_concentrated_siblings_leave(V, live, rejected, rest):
    """The residual's terms carry it, whatever the rejected ones were: a draw differs from the oracle's by a neighbour at most."""
    T, B, N, D = 0.25, 40, 8, 3
    live = np.array([v for v in live if v not in rejected])
    z = np.full((B, N, V), -np.inf, np.float32)
    z[:, :, live] = np.float32(T * np.log(rest / len(live)))
    z[:, :, list(rejected)] = np.float32(T) * np.log(np.array([1.0, 0.7, 0.3], np.float32))
    tok = np.zeros((B, N), np.int32)
    tok[:, 1:4] = rejected
    parent = np.tile(np.array([-1, 0, 0, 0, 0, 0, 0, 0], np.int32), (B, 1))
    u = np.full((B, 2 * N), 1.0 - 2.0 ** -24, np.float32)
    draws = np.concatenate([[0.0, 2.0 ** -24], np.random.default_rng(V).random(B - 2)]).astype(np.float32)
    u[:, N] = draws
    got = _accept(z, u, tok, parent, np.full(B, 4), D, T)
    # a term is exp of at most log(rest / n) / T: relative 2^-23 of the exponent twice, and of sums of 8192 terms in fixed trees of depth 13
    slack = 2.0 ** -22 * (abs(np.log(rest / len(live))) + 13)
    for b in range(B):
        cnt, path, ids, acc, (lo, hi) = po.accept_sampled(tok[b, :4], parent[b, :4], z[b, :4], T, u[b], n_max=N)
        assert list(got[b][0]) == [0] and list(path) == [0], "every sibling is rejected"
        at = int(np.searchsorted(live, got[b][1][0]))
        assert at < len(live) and live[at] == got[b][1][0], f"token {got[b][1][0]} has no mass"
        assert (at / len(live)) * (1 - slack) - slack <= draws[b] <= ((at + 1) / len(live)) * (1 + slack) + slack, (b, draws[b], at, ids)


def _candidates(z, K):
    """Per-128-logit candidates as the draft LM head leaves them: z [rows][Vd] fp32."""
    rows, Vd = z.shape
    tiles = (Vd + 127) // 128
    ld = sk.library().cand_pitch(tiles)
    val, idx = np.zeros((rows, ld, K), np.float32), np.full((rows, ld, K), -1, np.int32)
    mx, sm = np.full((rows, ld), -np.inf, np.float32), np.zeros((rows, ld), np.float32)
    for t in range(tiles):
        part = z[:, t * 128: (t + 1) * 128]
        order = np.argsort(-part, axis=1, kind="stable")[:, :K]
        n = order.shape[1]
        val[:, t, :n], idx[:, t, :n] = np.take_along_axis(part, order, 1), order + t * 128
        mx[:, t] = part.max(1)
        sm[:, t] = np.exp(part - part.max(1, keepdims=True)).sum(1)
    return val, idx, mx, sm, tiles


@pytest.mark.parametrize("levels", [2, 7, 0])                      # few distinct logits: more equal ones than the selections count; 0: all distinct
@pytest.mark.parametrize("K,Vd", [(1, 300), (4, 520), (6, 500), (10, 4100), (12, 2000)])
@pytest.mark.parametrize("which", [1, 2, 3])
def test_tree_step_targets_scores_and_skipped_sequences(which, K, Vd, levels):
    """Ids of the target vocabulary, scores, frontier, masks and inputs of the next pass, out of both selections; the middle sequence is
    skipped (what its rows hold is anything)."""
    B, D, k, half = 3, 3, 64, 8
    g = np.random.default_rng(which * 1000 + K + levels)
    rows = B * K
    z = (g.integers(0, levels, (rows, Vd)) / 4 if levels else g.standard_normal((rows, Vd))).astype(np.float32)
    val, idx, mx, sm, tiles = _candidates(z, K)
    val[K: 2 * K], mx[K: 2 * K] = np.nan, np.nan
    pool = K + (D - 1) * K * K
    d2t = g.permutation(3 * Vd)[:Vd].astype(np.int32)
    dev = lambda a, dt=torch.int32: torch.as_tensor(np.ascontiguousarray(a), dtype=dt).cuda()
    n, last = np.array([50, 60, 70]), np.array([0, -1, rows - 1])
    state = dev(np.stack([n, [1, 0, 1], last]))
    pool_i, score = dev(np.full((3, B, pool + 1), -9)), g.standard_normal((B, pool + 1)).astype(np.float32)
    front = np.full(B * D * K + 2 * B * K, -9, np.int32)
    frontier = front[: B * D * K].reshape(B, D, K)
    base = 0 if which == 1 else K + (which - 2) * K * K
    if which > 1:                                                  # the nodes this pass's rows stand for, of the level before
        lo = 1 if which == 2 else K + 1
        frontier[:, which - 1] = np.stack([lo + g.permutation(base + 1 - lo)[:K] for _ in range(B)])
    masks = g.integers(0, 2 ** 20, (2, rows)).astype(np.int64)
    x, embed = g.standard_normal((rows, k)).astype(np.float32), torch.randn(3 * Vd, k, generator=torch.Generator().manual_seed(K)).to(torch.bfloat16)
    score_d, front_d, masks_d, meta_d = dev(score, torch.float32), dev(front), dev(masks, torch.int64), dev(np.full((6, rows), -9))
    top, top_lp = dev(np.zeros(rows * K)), dev(np.zeros(rows * K), torch.float32)
    cat = torch.full((rows, 2 * k), 3.0, dtype=torch.bfloat16, device="cuda")
    inv_freq = 10.0 ** -np.arange(half)
    cs = torch.zeros(rows, half, 2, device="cuda")
    rc = sk.call("tree_step", state, pool_i, score_d, front_d, top, top_lp, meta_d, masks_d, dev(d2t), which, dev(val, torch.float32), dev(idx), dev(mx, torch.float32),
                 dev(sm, torch.float32), tiles, dev(x, torch.float32), embed.cuda(), cat, k, dev(inv_freq, torch.float64), cs, half, B, K, D)
    assert rc == 0, rc
    pool_i, score_o, front_o, masks_o, meta = (t.cpu().numpy() for t in (pool_i, score_d, front_d, masks_d, meta_d))
    fr_o, feat = front_o[: B * D * K].reshape(B, D, K), front_o[B * D * K + B * K:]
    for b in range(B):
        if b == 1:
            assert (pool_i[:, b] == -9).all() and np.array_equal(score_o[b], score[b])
            if which < D:
                assert not cat[b * K: (b + 1) * K].any() and (meta[0, b * K: (b + 1) * K] == -1).all()
            continue
        nrows = 1 if which == 1 else K
        child = []
        for r in range(nrows):
            row = last[b] if which == 1 else b * K + r
            par = 0 if which == 1 else frontier[b, which - 1, r]
            order = np.argsort(-z[row], kind="stable")[:K]
            lse = float(np.log(np.exp(z[row].astype(np.float64) - z[row].max()).sum()) + z[row].max())
            child += [(int(d2t[v]), int(par), float(score[b, par]) + float(z[row, v]) - lse, r) for v in order]
        at = slice(base + 1, base + 1 + len(child))
        assert [c[0] for c in child] == pool_i[0, b, at].tolist(), "target ids"
        assert [c[1] for c in child] == pool_i[1, b, at].tolist() and (pool_i[2, b, at] == which).all()
        assert np.abs(score_o[b, at] - [c[2] for c in child]).max() < 1e-5        # fp32 sums of up to 4100 terms, values of order 10
        if which == D:
            continue
        got = score_o[b, at]
        best = sorted(range(len(child)), key=lambda c: (-got[c], c))[:K]
        assert fr_o[b, which].tolist() == [base + 1 + c for c in best]
        for rr, c in enumerate(best):
            row, slot = b * K + rr, (which - 1) * K + rr
            src = last[b] if which == 1 else b * K + child[c][3]
            m = (0 if which == 1 else int(masks[0, src])) | 1 << slot
            assert feat[row] == src and int(masks_o[0, row]) == m
            assert meta[:, row].tolist() == [b, n[b] + which - 1, n[b] + slot, n[b], n[b], child[c][0]]
            assert torch.equal(cat[row].cpu(), torch.cat([torch.from_numpy(x[src]).to(torch.bfloat16), embed[child[c][0]]]))
            ang = (n[b] + which - 1) * inv_freq
            assert np.abs(cs[row].cpu().numpy() - np.stack([np.cos(ang), np.sin(ang)], 1)).max() < 1e-6


@pytest.mark.parametrize("K,D,N", [(2, 2, 4), (5, 3, 20), (6, 6, 60), (10, 5, 60), (10, 8, 64), (16, 4, 33)])
@pytest.mark.parametrize("levels", [1, 2, 5, 0])
def test_pruning_with_equal_scores_across_warps(K, D, N, levels):
    """The N - 1 best candidates, (score descending, pool index ascending), whichever side of a warp's own candidates the equal ones lie on."""
    pool, B = K + (D - 1) * K * K, 2
    g = np.random.default_rng(pool + levels)
    score, parent, depth = (np.zeros((B, pool + 1), dt) for dt in (np.float32, np.int32, np.int32))
    for b in range(B):
        front = [0]
        at = 1
        for d in range(1, D + 1):
            kids = []
            for f in front:
                for _ in range(K):
                    parent[b, at], depth[b, at] = f, d
                    # not above the parent's: a kept node's parent is kept
                    score[b, at] = score[b, f] - (g.integers(0, levels) if levels else g.random())
                    kids.append(at)
                    at += 1
            front = sorted(kids, key=lambda c: (-score[b, c], c))[:K]
    tok = g.integers(0, 1000, (B, pool + 1)).astype(np.int32)
    dev = lambda a, dt=torch.int32: torch.as_tensor(np.ascontiguousarray(a), dtype=dt).cuda()
    tree, nn, meta = dev(np.full((4, B, N), -9)), dev(np.zeros(B)), dev(np.full((6, B * N), -9))
    tscore, tmask, masks = torch.zeros(B, N, device="cuda"), dev(np.zeros((B, N)), torch.int64), dev(np.zeros((2, B * N)), torch.int64)
    assert sk.call("rerank", dev(np.stack([tok, parent, depth])), dev(score, torch.float32), dev(np.array([[30, 40], [1, 1]])), tree, tscore, tmask, nn, meta, masks, B, pool, N) == 0
    tree, nn = tree.cpu().numpy(), nn.cpu().numpy()
    M = min(N - 1, pool)
    for b in range(B):
        kept = [0] + sorted(sorted(range(1, pool + 1), key=lambda c: (-score[b, c], c))[:M])
        assert nn[b] == M + 1 and tree[3, b, : M + 1].tolist() == kept
        assert tree[0, b, : M + 1].tolist() == tok[b, kept].tolist()
        assert tree[1, b, : M + 1].tolist() == [-1] + [kept.index(int(parent[b, c])) for c in kept[1:]]
