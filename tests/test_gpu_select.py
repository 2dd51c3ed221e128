"""The selection of a round as integer work: the mask must hold the R smallest (score bits, index) of the scores
that the same call returns, and the compaction must move every slot accordingly.  Sizes cover the fused and the
separate finalize, one to eight CTAs per unit, keys that do not fit a CTA's shared memory, and ties at the cutoff."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# KV heads, slots, keys repeated every `period` slots (0: none; with it most scores occur many times)
@pytest.mark.parametrize("hkv,n,period,first_round", [
    (2, 300, 0, 0), (3, 8200, 0, 1), (3, 8400, 64, 0), (8, 20011, 128, 1), (2, 140000, 0, 0), (2, 140000, 512, 1),
    (160, 66200, 512, 0),
    # one kernel and two, few units and many, around 1024 to 4096 pairs
    (50, 2084, 0, 0), (50, 2086, 32, 0), (17, 5212, 0, 0), (17, 5214, 32, 1), (16, 6181, 64, 1), (16, 6184, 0, 1),
    (128, 8228, 64, 0), (128, 8230, 0, 0)])
def test_mask_is_the_smallest_scores(hkv, n, period, first_round):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(n + period)
    K, V = (torch.empty(1, hkv, n, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for x in (K, V):
        rows = torch.randn(hkv, period or n, 128, generator=g, device="cuda").to(torch.bfloat16)
        x[0] = rows.repeat(1, n // (period or n) + 1, 1)[:, :n]
    counts = torch.ones(1, hkv, n, dtype=torch.int32, device="cuda")
    q = torch.randn(1, hkv, 4, 128, generator=g, device="cuda").to(torch.bfloat16)
    p = kb.make_params(K, V, hkv, 4, causal=False, first_round=first_round)
    ws = torch.empty(kb.kvs_workspace_size(p, n, 0), dtype=torch.uint8, device="cuda")
    score, w = (torch.zeros(1, hkv, n // 2, device="cuda") for _ in range(2))
    mask = torch.zeros(1, hkv, n // 2, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    _, off, P, R = kb.kvs_round_plan(p, n, n - n // 5)[0]
    kb.kvs_window_stats(p, K, V, counts, q, [n], [n - n // 5], ws, score=score, w=w, mask=mask, status_dev=status)
    want = torch.zeros_like(mask)
    order = torch.sort(score[0, :, :P], dim=-1, stable=True).indices[:, :R]
    want[0].scatter_(1, order, 1)
    assert torch.equal(mask, want)
    if period:
        cut = score[0].gather(1, order[:, -1:])
        assert int((score[0, :, :P] == cut).sum(1).min()) > 1       # the cutoff is a tie
    # the same decision through kvs_compact: the map counts the merged pairs before every slot
    index = torch.zeros(1, hkv, n, dtype=torch.int32, device="cuda")
    kb.kvs_compact(p, K, V, counts, mask, w, [n], [R], ws, new_index=index, status_dev=status)
    before = torch.zeros(hkv, n, dtype=torch.int32, device="cuda")
    before[:, off + 1:off + 2 * P:2] = want[0, :, :P].int()          # the right member of a merged pair moves up by one
    slots = torch.arange(n, dtype=torch.int32, device="cuda")
    assert torch.equal(index[0], slots - before.cumsum(1, dtype=torch.int32))
    assert status.item() == 0


# KV heads, slots, period of the keys, factor of the queries.  Large queries leave most slots with masses far below 2^-56
# or of 0, whose scores share the first bin of the first pass, so that all four passes are needed; a period of 2 gives all pairs
# one score, and every pass goes on until the interval is that one pattern; the last cases walk more than 32 steps a CTA.
@pytest.mark.parametrize("hkv,n,period,factor", [
    (2, 300, 2, 1), (2, 2200, 2, 1), (3, 2200, 0, 30), (8, 2084, 0, 4), (3, 8400, 16, 1), (8, 40001, 0, 30), (8, 40001, 2, 1),
    (2, 140000, 64, 1), (160, 66200, 0, 30), (160, 66200, 2, 1)])
def test_a_pass_takes_the_smallest_scores(hkv, n, period, factor):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(n + period + factor)
    K, V = (torch.empty(1, hkv, n, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for x in (K, V):
        rows = torch.randn(hkv, period or n, 128, generator=g, device="cuda").to(torch.bfloat16)
        x[0] = rows.repeat(1, n // (period or n) + 1, 1)[:, :n]
    counts = torch.ones(1, hkv, n, dtype=torch.int32, device="cuda")
    q = (factor * torch.randn(1, hkv, 4, 128, generator=g, device="cuda")).to(torch.bfloat16)
    p = kb.make_params(K, V, hkv, 4, causal=False)
    ws = torch.empty(kb.kvs_workspace_size(p, n, 0), dtype=torch.uint8, device="cuda")
    score, w = (torch.zeros(1, hkv, n // 2, device="cuda") for _ in range(2))
    mask = torch.zeros(1, hkv, n // 2, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    _, off, P, R = kb.kvs_round_plan(p, n, n - n // 5)[0]
    kb.kvs_window_stats(p, K, V, counts, q, [n], [n - n // 5], ws, score=score, w=w, mask=mask, status_dev=status)
    want = torch.zeros_like(mask)
    want[0].scatter_(1, torch.sort(score[0, :, :P], dim=-1, stable=True).indices[:, :R], 1)
    assert torch.equal(mask, want)
    # one round of a pass makes the same decision and counts its tiles alike
    K2, V2, counts2 = K.clone(), V.clone(), counts.clone()
    kb.kvs_compact(p, K2, V2, counts2, mask, w, [n], [R], ws, status_dev=status)
    assert kb.kvs_merge_layer(p, K, V, counts, q, [n], [n - R], ws, status_dev=status) == [n - R]
    for x, y in ((K, K2), (V, V2), (counts, counts2)):
        assert torch.equal(x[:, :, :n - R].view(torch.int16 if x is not counts else torch.int32),
                           y[:, :, :n - R].view(torch.int16 if x is not counts else torch.int32))
    assert status.item() == 0


# KV heads, slots, pairs, bits of a key channel.  Both sides of the lines between one kernel and two.  A long protected suffix leaves few pairs (one kernel adds the partials and
# selects, with and without a CTA to an SM) but more steps of a warp than keys are kept; with undefined keys every score is
# NaN, of either sign as the sums may have it, and the first pairs are taken.
@pytest.mark.parametrize("hkv,n,pairs,bits", [(17, 3200, 1536, None), (17, 3200, 1537, None), (16, 6300, 3072, None), (16, 6300, 3073, None),
                                              (150, 3200, 1536, None), (150, 3200, 1537, None), (2, 80000, 2000, None), (150, 70000, 600, None), (2, 2200, 1000, 0x7FC0), (2, 2200, 1000, 0xFFC0),
                                              (3, 9000, 4400, 0xFFC0), (150, 1400, 650, 0x7FC0), (2, 80000, 2000, 0xFFC0),
                                              (2, 300000, 149000, 0xFFC0)])
def test_steps_beyond_the_kept_keys_and_undefined_scores(hkv, n, pairs, bits):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(n + pairs)
    K, V = (torch.randn(1, hkv, n, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    if bits is not None:
        K.view(torch.int16)[0, :, 40, 7] = bits - (1 << 16 if bits >> 15 else 0)
    counts = torch.ones(1, hkv, n, dtype=torch.int32, device="cuda")
    q = torch.randn(1, hkv, 4, 128, generator=g, device="cuda").to(torch.bfloat16)
    p = kb.make_params(K, V, hkv, 4, causal=False, recent=n - 32 - 2 * pairs)
    ws = torch.empty(kb.kvs_workspace_size(p, n, 0), dtype=torch.uint8, device="cuda")
    score, w = (torch.zeros(1, hkv, n // 2, device="cuda") for _ in range(2))
    mask = torch.zeros(1, hkv, n // 2, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    budget = n - pairs // 3
    _, off, P, R = kb.kvs_round_plan(p, n, budget)[0]
    assert P == pairs and R == pairs // 3
    kb.kvs_window_stats(p, K, V, counts, q, [n], [budget], ws, score=score, w=w, mask=mask, status_dev=status)
    key = score[0, :, :P].view(torch.int32)
    assert int(key.min()) >= 0
    assert bits is None or bool(torch.isnan(score[0, :, :P]).all())
    want = torch.zeros_like(mask)
    want[0].scatter_(1, torch.sort(key, dim=-1, stable=True).indices[:, :R], 1)
    assert torch.equal(mask, want) and status.item() == 0
    # the counts in front of the tiles, the empty ones of the suffix among them
    index = torch.zeros(1, hkv, n, dtype=torch.int32, device="cuda")
    kb.kvs_compact(p, K, V, counts, mask, w, [n], [R], ws, new_index=index, status_dev=status)
    before = torch.zeros(hkv, n, dtype=torch.int32, device="cuda")
    before[:, off + 1:off + 2 * P:2] = want[0, :, :P].int()
    assert torch.equal(index[0], torch.arange(n, dtype=torch.int32, device="cuda") - before.cumsum(1, dtype=torch.int32))
    assert status.item() == 0
