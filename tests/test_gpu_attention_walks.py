"""The attention kernel's stabiliser is the maximum over a CTA's first tile of 128 slots.  Rows whose later logits
are larger by a little, by almost and by more than the range of an exponent of a part of the sum allows (2^60: the
CTA then walks its slots again with the true maxima), and rows whose first tiles are negligible, against the oracle.
The first test has few units, whose slots are cut into ranges of one tile each (each with its own stabiliser); the others
have so many that a CTA walks eight or nine tiles.

P' carries 16 significant bits and is at most 2^60 times the first tile's largest: the relative error of an
output stays 2^-17 max |V / c|, below 1e-4 here, plus the fp32 error of a logit of up to 320 (2^-24 * 320 = 2e-5,
times |V|)."""
import numpy as np
import pytest

from oracle import kvs_oracle as oc
from paper_2603_00907_b200 import workloads as wl
from tests import kvs_testlib as tl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,spikes", [(640, {600: 30.0}), (640, {130: 45.0, 639: 60.0}), (900, {500: 100.0}),
                                      (900, {0: 90.0}), (3000, {127: 20.0, 128: 150.0, 2999: 300.0}), (129, {128: 220.0})])
def test_later_slots_outgrow_the_first_tile(n, spikes):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    hq, hkv, t = 8, 2, 40                                 # 160 query rows per KV head: two query blocks
    w = wl.small_case(seed=n, n_q_heads=hq, n_kv_heads=hkv, window=8, seq_lens=(n,), budgets=(n,), n_decode=t)
    data = wl.make_layer(w)
    rng = np.random.default_rng(n)
    # queries share a direction, so that a key along it has about the wanted logit for every one of them
    u = rng.standard_normal(128)
    u /= np.linalg.norm(u)
    q = 0.05 * rng.standard_normal((1, hq, t, 128)) + 8.0 * u
    data["q_new"] = wl.f32_to_bf16_bits(q.astype(np.float32))
    data["counts"][:] = rng.integers(1, 5, size=data["counts"].shape)
    for j, logit in spikes.items():
        data["K"][0, :, j] = wl.f32_to_bf16_bits((logit * np.sqrt(128.0) / 8.0 * u).astype(np.float32))
    dev = tl.upload_layer(data)
    p = kb.make_params(dev["K"], dev["V"], hq, 8)
    ws = torch.empty(kb.kvs_workspace_size(p, n, t), dtype=torch.uint8, device="cuda")
    out = torch.zeros((1, hq, t, 128), dtype=torch.bfloat16, device="cuda")
    lse = torch.zeros((1, hq, t), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        kb.kvs_decode_attn(p, dev["q_new"], dev["K"], dev["V"], dev["counts"], [n], out, ws, lse=lse, status_dev=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    og, lg, G = tl.bits_of(out), lse.cpu().numpy(), hq // hkv
    for h in range(hkv):
        hs = slice(h * G, (h + 1) * G)
        ref, lse_ref = oc.decode_attention(data["q_new"][0, hs], data["K"][0, h, :n], data["V"][0, h, :n],
                                           data["counts"][0, h, :n])
        ok, mx, _, _ = tl.bf16_close(og[0, hs], oc.f64_to_bf16(ref), atol=2e-4)
        assert ok, (h, mx)
        assert np.max(np.abs(lg[0, hs] - lse_ref)) < 1e-4 * max(1.0, np.max(np.abs(lse_ref)) / 20)


# Ranges of many tiles.  With 80 heads of one query block (or two, for the window pass) the GPU has no idle SM to cut a head's
# slots for, and one CTA walks them all: 8 or 9 tiles of 128 here.  A logit of 100 is 2^144 above the first
# tile's: without the walks with true maxima its weight would be infinite and its row NaN.
LATE = [(1000, {150: 30.0, 700: 38.0}), (1000, {200: 41.0, 640: 44.0, 999: 43.0}), (1000, {999: 100.0}),
        (1100, {128: 90.0, 129: 150.0, 1099: 300.0}), (1030, {700: 120.0}), (1100, {5: 60.0, 300: 200.0})]


def _spiked(n, spikes, q_shape, seed):
    """Keys, values and queries whose logit at the slots of `spikes` is about the given one for every query; the keys and
    values of 50 slots behind the n hold NaN."""
    hkv = 80
    rng = np.random.default_rng(seed)
    w = wl.small_case(seed=seed, n_q_heads=hkv, n_kv_heads=hkv, window=8, seq_lens=(n + 50,), budgets=(n,))
    data = wl.make_layer(w)
    u = rng.standard_normal(128)
    u /= np.linalg.norm(u)
    data["q"] = wl.f32_to_bf16_bits((0.05 * rng.standard_normal(q_shape) + 8.0 * u).astype(np.float32))
    data["counts"][:] = rng.integers(1, 5, size=data["counts"].shape)
    for j, logit in spikes.items():
        data["K"][0, :, j] = wl.f32_to_bf16_bits((logit * np.sqrt(128.0) / 8.0 * u).astype(np.float32))
    data["K"][0, :, n:] = 0x7FC0
    data["V"][0, :, n:] = 0x7FC0
    return data


@pytest.mark.parametrize("n,spikes", LATE)
def test_later_tiles_of_a_long_range_outgrow_the_first(n, spikes):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    hkv, t = 80, 40
    data = _spiked(n, spikes, (1, hkv, t, 128), n)
    K, V, q = (tl.to_dev_bf16(data[k]) for k in ("K", "V", "q"))
    counts = torch.from_numpy(data["counts"]).cuda()
    p = kb.make_params(K, V, hkv, 8)
    ws = torch.empty(kb.kvs_workspace_size(p, n + 50, t), dtype=torch.uint8, device="cuda")
    out = torch.zeros((1, hkv, t, 128), dtype=torch.bfloat16, device="cuda")
    lse = torch.zeros((1, hkv, t), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        kb.kvs_decode_attn(p, q, K, V, counts, [n], out, ws, lse=lse, status_dev=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    og, lg = tl.bits_of(out), lse.cpu().numpy()
    for h in (0, 33, 79):
        ref, lse_ref = oc.decode_attention(data["q"][0, h:h + 1], data["K"][0, h, :n], data["V"][0, h, :n], data["counts"][0, h, :n])
        ok, mx, _, _ = tl.bf16_close(og[0, h:h + 1], oc.f64_to_bf16(ref), atol=2e-4)
        assert ok, (h, mx)
        assert np.max(np.abs(lg[0, h:h + 1] - lse_ref)) < 1e-4 * max(1.0, np.max(np.abs(lse_ref)) / 20)


@pytest.mark.parametrize("n,spikes", LATE)
@pytest.mark.parametrize("window,first_round", [(24, 0), (24, 1), (130, 1)])
def test_window_pass_with_pair_norms_walks_again(n, spikes, window, first_round):
    """The same in the window pass, with one query block and with two, tiles aligned with the pairs of either parity, the
    causal mask, and the pair-norm warps handing the stages of the further walks back."""
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    hkv = 80
    spikes = {j: v for j, v in spikes.items() if j < n - window}      # (the last slots are hidden from the first queries)
    data = _spiked(n, spikes, (1, hkv, window, 128), n + window)
    K, V, q = (tl.to_dev_bf16(data[k]) for k in ("K", "V", "q"))
    counts = torch.from_numpy(data["counts"]).cuda()
    p = kb.make_params(K, V, hkv, window, first_round=first_round)
    n_max = n + 50
    ws = torch.empty(kb.kvs_workspace_size(p, n_max, 0), dtype=torch.uint8, device="cuda")
    A, N1 = torch.zeros(1, hkv, n_max, device="cuda"), torch.zeros(1, hkv, n_max, device="cuda")
    cosv = torch.zeros(1, hkv, n_max // 2, device="cuda")
    o, lse = torch.zeros(1, hkv, window, 128, device="cuda"), torch.zeros(1, hkv, window, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    kb.kvs_window_stats(p, K, V, counts, q, [n], [n - 100], ws, A=A, N1=N1, cosv=cosv, o_win=o, lse_win=lse, status_dev=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    for h in (0, 41, 79):
        st = oc.round_stats(data["K"][0, h, :n], data["V"][0, h, :n], data["counts"][0, h, :n].astype(np.int64),
                            data["q"][0, h:h + 1], n - 100, first_round, window=window, sink=32, recent=window,
                            scale=1 / np.sqrt(128.0), causal=True, round_frac=0.5, score_mode=0)
        off, P = st["off"], st["P"]
        ok, ratio, _ = tl.stat_close(o[0, h].cpu().numpy(), st["o"], rtol=2e-4)      # (P' may be 2^60 times the first tile's)
        assert ok, (h, ratio)
        # the fp32 error of a logit, 2^-22 of it, is a relative error of its weight
        rtol = tl.STAT_RTOL + 2.0 ** -22 * max(spikes.values(), default=0.0)
        sl = np.arange(off, off + 2 * P)
        ok, ratio, _ = tl.rel_close(A[0, h].cpu().numpy()[sl], st["A"][sl], rtol=rtol)
        assert ok, (h, ratio)
        assert np.max(np.abs(cosv[0, h, :P].cpu().numpy() - st["cos"])) <= tl.COS_ATOL
        # (a slot that has a row to itself is the row's output: its distance from it is rounding)
        far = sl[~np.isin(sl, list(spikes))]
        ok, ratio, _ = tl.rel_close(N1[0, h].cpu().numpy()[far], st["N1"][far], rtol=2 * rtol)
        assert ok, (h, ratio)
