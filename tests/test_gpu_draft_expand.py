"""CUDA draft step (through the C ABI) against the oracle: tokens, parents, joint values (one fp32
addition) and the next frontier, all bit-exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_15562_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _check(ctx, lp, flp, fc, k, width, base, cap):
    B = lp.shape[0]
    ref = [np.full((B, cap), -7, np.int32), np.full((B, cap), -7, np.int32), np.full((B, cap), -3.5, np.float32)]
    nc_ref, nl_ref = oracle.draft_expand(lp, flp, fc, k, width, base, *ref)
    got = [_dev(np.full((B, cap), -7, np.int32)), _dev(np.full((B, cap), -7, np.int32)),
           _dev(np.full((B, cap), -3.5, np.float32))]
    nc, nl = ctx.draft_expand(_dev(lp), _dev(flp), _dev(fc), k, width, base, *got)
    ctx.check()
    for g, r in zip(got, ref):
        assert np.array_equal(g.cpu().numpy(), r)            # new entries equal, all others untouched
    assert np.array_equal(nc.cpu().numpy(), nc_ref)
    assert np.array_equal(nl.cpu().numpy(), nl_ref)


@pytest.mark.parametrize("vocab", [17, 1000, 4099, 32000, 128256])
@pytest.mark.parametrize("step", [0.0, 0.5])
def test_vocab_sizes_and_ties(vocab, step):
    """Rows shorter than one piece, ragged last pieces, unaligned row starts (odd vocab), 32 pieces."""
    ctx = binding.Context(8, 2, vocab, 256, max_nodes=64, max_batch=4)
    rng = np.random.default_rng(vocab)
    for seed, (F, k, width) in enumerate([(1, 10, 10), (10, 10, 10), (16, 16, 16), (3, 5, 15)]):
        if k > vocab:
            continue
        B = 2
        lp = synth.draft_logprob_rows(seed, B, F, vocab, step=step)
        flp = (-rng.random((B, F)) * 4).astype(np.float32)
        fc = rng.integers(-1, 50, size=(B, F)).astype(np.int32)
        _check(ctx, lp, flp, fc, k, width, 50, 50 + F * k + 3)


def test_minus_infinity_rows_and_zero_values():
    vocab = 5000
    ctx = binding.Context(8, 2, vocab, 256, max_nodes=64, max_batch=2)
    lp = synth.draft_logprob_rows(1, 2, 4, vocab)
    lp[0, 0, :] = -np.inf                       # impossible everywhere: tokens 0 .. k-1 by index
    lp[0, 1, 10:] = -np.inf                     # fewer finite values than k
    lp[1, 2, 77] = 0.0
    lp[1, 2, 78] = -0.0                         # the two zeros are one value: the lower token first
    flp = np.zeros((2, 4), np.float32)
    fc = np.full((2, 4), -1, np.int32)
    _check(ctx, lp, flp, fc, 12, 7, 0, 48)


def test_whole_draft_phase_then_builder_matches_the_oracle_chain():
    """Five levels of top-10 expansion on the device, then the builder: the flattened 60-node tree
    equals the one the oracle derives from the same log-probability rows."""
    B, V, k, width, levels, N = 2, 32000, 10, 10, 5, 60
    cap = k + (levels - 1) * width * k
    ctx = binding.Context(8, 2, V, 256, max_nodes=N, max_batch=B)
    ref = [np.full((B, cap), -7, np.int32), np.full((B, cap), -7, np.int32), np.full((B, cap), 0, np.float32)]
    dev = [_dev(a.copy()) for a in ref]
    fc_r, fl_r = np.full((B, 1), -1, np.int32), np.zeros((B, 1), np.float32)
    fc_d, fl_d = _dev(fc_r), _dev(fl_r)
    base = 0
    for lvl in range(levels):
        F = fc_r.shape[1]
        lp = synth.draft_logprob_rows(300 + lvl, B, F, V)
        fc_r, fl_r = oracle.draft_expand(lp, fl_r, fc_r, k, min(width, F * k), base, *ref)
        fc_d, fl_d = ctx.draft_expand(_dev(lp), fl_d, fc_d, k, min(width, F * k), base, *dev)
        base += F * k
    root = np.array([5, 6], np.int32)
    want = oracle.tree_build(*ref, root, N)
    parent, token, cand, n_out = ctx.tree_build(*dev, _dev(root), N)
    ctx.check()
    assert want["valid"]
    assert np.array_equal(parent.cpu().numpy(), want["parent"])
    assert np.array_equal(token.cpu().numpy(), want["token"])
    assert np.array_equal(cand.cpu().numpy(), want["cand"])


def test_host_detected_errors():
    ctx = binding.Context(8, 2, 1000, 256, max_nodes=64, max_batch=1)
    lp = _dev(synth.draft_logprob_rows(0, 1, 2, 1000))
    args = (_dev(np.zeros((1, 2), np.float32)), _dev(np.full((1, 2), -1, np.int32)))
    arrs = [_dev(np.zeros((1, 8), np.int32)), _dev(np.zeros((1, 8), np.int32)), _dev(np.zeros((1, 8), np.float32))]
    with pytest.raises(binding.FspadError):
        ctx.draft_expand(lp, *args, 5, 4, 0, *arrs)          # 2 * 5 new candidates do not fit 8 entries
    with pytest.raises(binding.FspadError):
        ctx.draft_expand(lp, *args, 17, 4, 0, *arrs)         # top_k beyond 16
    with pytest.raises(binding.FspadError):
        ctx.draft_expand(lp, *args, 2, 5, 0, *arrs)          # width beyond the new candidates


@pytest.mark.parametrize("vocab,batch,F,k,width", [(4095, 1, 1, 16, 16), (4096, 1, 16, 16, 40), (4097, 2, 3, 1, 3), (8193, 1, 2, 4, 8),
                                                   (50257, 16, 10, 10, 10), (128256, 16, 16, 16, 256), (128256, 1, 1, 10, 10)])
@pytest.mark.parametrize("order", ["random", "ascending", "constant"])
def test_piece_lengths_and_long_lists(vocab, batch, F, k, width, order):
    """One to sixteen pieces per row of one or several rounds of 4096 tokens, row starts at every alignment; ascending rows (every
    token of a later round reaches the first round's bound, so the lists have to be cut) and constant ones (all are ties)."""
    ctx = binding.Context(8, 2, vocab, 256, max_nodes=64, max_batch=batch)
    rng = np.random.default_rng(vocab + F)
    lp = rng.standard_normal((batch, F, vocab), dtype=np.float32)
    if order == "ascending":
        lp.sort(-1)
    elif order == "constant":
        lp[:] = -2.5
    flp = rng.standard_normal((batch, F)).astype(np.float32)
    fc = rng.integers(0, 5, (batch, F)).astype(np.int32)
    for _ in range(2):                                       # the counters are back at zero after a call
        _check(ctx, lp, flp, fc, k, width, 7, 7 + F * k)


@pytest.mark.parametrize("batch,F,k,width", [(1, 1, 10, 10), (16, 1, 10, 10), (16, 10, 10, 4), (16, 4, 8, 9), (16, 10, 10, 10), (7, 16, 16, 16)])
@pytest.mark.parametrize("shift", [0, 4])
def test_next_frontier_over_the_current_one(batch, F, k, width, shift):
    """The frontier's buffers used for the next one as well, in place or a few entries further: every sequence still starts from its own
    current frontier, whichever sequence finishes first."""
    vocab = 20000
    ctx = binding.Context(8, 2, vocab, 256, max_nodes=64, max_batch=batch)
    rng = np.random.default_rng(F * 31 + width)
    lp = rng.standard_normal((batch, F, vocab), dtype=np.float32)
    flp = rng.standard_normal((batch, F)).astype(np.float32)
    fc = rng.integers(0, 50, (batch, F)).astype(np.int32)
    cap = 60 + F * k
    ref = [np.full((batch, cap), -7, np.int32), np.full((batch, cap), -7, np.int32), np.full((batch, cap), -3.5, np.float32)]
    nc_ref, nl_ref = oracle.draft_expand(lp, flp, fc, k, width, 60, *ref)
    dlp, room = _dev(lp), batch * max(F, width) + shift
    for _ in range(3):
        bufs = torch.zeros(room, dtype=torch.int32, device="cuda"), torch.zeros(room, dtype=torch.float32, device="cuda")
        cand, logp = (t[:batch * F].view(batch, F) for t in bufs)
        nxt = tuple(t[shift:shift + batch * width].view(batch, width) for t in bufs)
        cand.copy_(_dev(fc))
        logp.copy_(_dev(flp))
        got = [_dev(np.full((batch, cap), -7, np.int32)), _dev(np.full((batch, cap), -7, np.int32)),
               _dev(np.full((batch, cap), -3.5, np.float32))]
        ctx.draft_expand(dlp, logp, cand, k, width, 60, *got, *nxt)
        ctx.check()
        for g, r in zip(got, ref):
            assert np.array_equal(g.cpu().numpy(), r)
        assert np.array_equal(nxt[0].cpu().numpy(), nc_ref) and np.array_equal(nxt[1].cpu().numpy(), nl_ref)


@pytest.mark.parametrize("vocab,batch,F", [
    (151937, 1, 10),       # 14 pieces: one CTA per SM
    (36865, 1, 14),        # ten pieces, the last one shorter
    (50257, 4, 10),        # seven pieces of two rounds
    (20003, 16, 10),       # three pieces, four CTAs per SM
    (20003, 16, 16),       # two pieces, four CTAs per SM
    (32003, 16, 16),       # the same with longer ones
])
def test_pieces_by_rows_and_vocabulary(vocab, batch, F):
    ctx = binding.Context(8, 2, vocab, 256, max_nodes=64, max_batch=batch)
    rng = np.random.default_rng(vocab + batch)
    lp = np.round(rng.standard_normal((batch, F, vocab), dtype=np.float32) * 3, 2)      # with ties
    flp = rng.standard_normal((batch, F)).astype(np.float32)
    fc = rng.integers(0, 5, (batch, F)).astype(np.int32)
    _check(ctx, lp, flp, fc, 10, 10, 7, 7 + F * 10)


@pytest.mark.parametrize("more", [0, 22, 23, 118, 119, 502, 503, 4598, 4599])
@pytest.mark.parametrize("values", ["apart", "equal"])
@pytest.mark.parametrize("k,width", [(10, 32), (10, 33), (16, 16)])
def test_lengths_of_a_piece_s_list(more, values, k, width):
    """A row's list takes the tokens that reach the k-th largest half-warp maximum of its first 4096: k of those and `more` behind them,
    on either side of what a warp ranks as it is (32), cuts first (128), what is kept between rounds (512) and what there is room for."""
    V, F, B = 16384, 16, 8
    ctx = binding.Context(8, 2, V, 256, max_nodes=64, max_batch=B)
    rng = np.random.default_rng(more)
    lp = np.full((B, F, V), -50.0, np.float32)
    lp[:, :, :4096:4096 // 32][:, :, :k] = -10.0                 # tokens 0, 128, ...: one for each of k half-warps
    for b in range(B):
        for f in range(F):
            at = 4096 + rng.choice(V - 4096, more, replace=False)
            lp[b, f, at] = -10.0 if values == "equal" else -10.0 + 9.0 * rng.random(more, dtype=np.float32)
    flp = (-rng.random((B, F)) * 4).astype(np.float32)
    fc = rng.integers(-1, 50, size=(B, F)).astype(np.int32)
    _check(ctx, lp, flp, fc, k, width, 0, F * k)


@pytest.mark.parametrize("vocab", [4096, 4097, 16385, 32000])
@pytest.mark.parametrize("above", [0, 9, 15, 16, 20, 40])
@pytest.mark.parametrize("k", [10, 16])
def test_many_equal_values(vocab, above, k):
    """Rows of one value, with a few tokens above it (of one value, or of two): what a warp's bound does not shorten is cut by a search
    over tokens alone where fewer than k lie above the lowest value, by values and tokens elsewhere."""
    F, B = 10, 3
    ctx = binding.Context(8, 2, vocab, 256, max_nodes=64, max_batch=B)
    rng = np.random.default_rng(vocab + above)
    lp = np.full((B, F, vocab), -9.0, np.float32)
    for b in range(B):
        for f in range(F):
            at = rng.choice(vocab, above, replace=False)
            lp[b, f, at] = -8.0
            if f % 2:
                lp[b, f, at[:above // 3]] = -7.5
    flp = (-rng.random((B, F)) * 4).astype(np.float32)
    fc = rng.integers(-1, 50, size=(B, F)).astype(np.int32)
    _check(ctx, lp, flp, fc, k, k, 0, F * k)
