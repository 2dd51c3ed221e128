"""Infinite and undefined logits.  A key with an infinite channel gives its slot a logit of -inf, i.e. no weight, wherever
in a sequence such slots stand; a key with a NaN makes the rows that see it NaN; neither may be lost or spread when
the parts of a row (blocks, warps, CTAs, key ranges) are merged.  Against the oracle in float64.

Finite outputs are held to what P' in 16 significant bits gives, 2^-17 max |V| < 1e-4 before the bf16 rounding; the
log-sum-exp to the fp32 error of a logit, 3e-6 of values below 20 (1e-4 with the sum's) and in proportion above."""
import numpy as np
import pytest

from oracle import kvs_oracle as oc
from paper_2603_00907_b200 import workloads as wl
from tests import kvs_testlib as tl

pytestmark = pytest.mark.gpu

NEG_INF, NAN = 0xFF80, 0x7FC0


def _attend(hq, hkv, t, n, low=(), nan=(), edit=None, every=1):
    """Decode attention of `t` tokens over n slots whose logits are -inf in the ranges `low` and NaN in `nan`;
    checked against the oracle for every KV head (or every `every`-th)."""
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    w = wl.small_case(seed=n + t, n_q_heads=hq, n_kv_heads=hkv, window=8, seq_lens=(n,), budgets=(n,), n_decode=t)
    data = wl.make_layer(w)
    data["q_new"][..., 0] = 0x3F80                        # 1.0: an infinite key channel 0 decides the logit
    for lo, hi in low:
        data["K"][0, :, lo:hi, 0] = NEG_INF
    for lo, hi in nan:
        data["K"][0, :, lo:hi, 5] = NAN
    if edit:
        edit(data)
    dev = tl.upload_layer(data)
    p = kb.make_params(dev["K"], dev["V"], hq, 8)
    ws = torch.empty(kb.kvs_workspace_size(p, n, t), dtype=torch.uint8, device="cuda")
    out = torch.zeros((1, hq, t, 128), dtype=torch.bfloat16, device="cuda")
    lse = torch.zeros((1, hq, t), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    kb.kvs_decode_attn(p, dev["q_new"], dev["K"], dev["V"], dev["counts"], [n], out, ws, lse=lse, status_dev=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    if nan:
        assert torch.isnan(out).all() and torch.isnan(lse).all()
        return
    og, lg, G = tl.bits_of(out), lse.cpu().numpy(), hq // hkv
    for h in range(0, hkv, every):
        hs = slice(h * G, (h + 1) * G)
        ref, lse_ref = oc.decode_attention(data["q_new"][0, hs], data["K"][0, h, :n], data["V"][0, h, :n],
                                           data["counts"][0, h, :n])
        ok, mx, _, _ = tl.bf16_close(og[0, hs], oc.f64_to_bf16(ref), atol=1e-4)
        assert ok, (h, mx)
        assert np.max(np.abs(lg[0, hs] - lse_ref)) < 1e-4 * max(1.0, np.max(np.abs(lse_ref)) / 20)


# 4, 8 and 16 rows; one CTA, one cluster, several clusters per unit
FEW_ROWS = [(4, 1, 1, 200), (4, 1, 1, 6000), (8, 1, 1, 640), (1, 1, 7, 6200), (8, 2, 4, 1500)]


@pytest.mark.parametrize("hq,hkv,t,n", FEW_ROWS)
@pytest.mark.parametrize("low", [((0, 16),), ((0, 130),), ((16, 48), (64, 96)), ((3, None),)])
def test_few_rows_with_slots_of_no_weight(hq, hkv, t, n, low):
    _attend(hq, hkv, t, n, low=[(lo, n if hi is None else hi) for lo, hi in low])


@pytest.mark.parametrize("hq,hkv,t,n", FEW_ROWS)
@pytest.mark.parametrize("nan", [(0, 16), (16, 32), (128, 200), (7, 8), (0, None)])
def test_few_rows_that_see_a_nan(hq, hkv, t, n, nan):
    _attend(hq, hkv, t, n, nan=[(nan[0], n if nan[1] is None else nan[1])])


# more than 16 rows: ranges of one, three, six, 24 and 3 tiles of 128 slots; a combine of few rows and of many; the last
# without padding rows in its block of 128 (zero queries, whose product with an infinite key is NaN)
MANY_ROWS = [(2, 2, 20, 700), (64, 64, 24, 700), (90, 90, 40, 700), (80, 80, 40, 3000), (64, 64, 128, 700)]


@pytest.mark.parametrize("hq,hkv,t,n", MANY_ROWS)
@pytest.mark.parametrize("nan", [(300, 301), (0, 128), (640, 700), (0, None)])
def test_many_rows_that_see_a_nan(hq, hkv, t, n, nan):
    _attend(hq, hkv, t, n, nan=[(nan[0], n if nan[1] is None else nan[1])])


@pytest.mark.parametrize("hq,hkv,t,n", FEW_ROWS)
@pytest.mark.parametrize("slot", [0, 5, 130])
def test_few_rows_whose_largest_weight_has_an_infinite_value(hq, hkv, t, n, slot):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    q, K, V = (torch.randn(1, h, m, 128, generator=g, device="cuda").to(torch.bfloat16) for h, m in ((hq, t), (hkv, n), (hkv, n)))
    q[..., 0], K[..., 0], K[:, :, slot, 0] = 8.0, 0.0, 20.0   # a logit of 14 against 0 +- 1
    V[:, :, slot] = float("inf")
    counts = torch.ones(1, hkv, n, dtype=torch.int32, device="cuda")
    p = kb.make_params(K, V, hq, 8)
    ws = torch.empty(kb.kvs_workspace_size(p, n, t), dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(q)
    kb.kvs_decode_attn(p, q, K, V, counts, [n], out, ws)
    assert (out == float("inf")).all()


def _rest_far_below(lo):
    """Keys from slot lo on with logits of about -265 (e to that power is no float)."""
    def edit(data):
        data["K"][0, :, lo:, 0] = wl.f32_to_bf16_bits(np.float32([-3000.0]))[0]
    return edit


@pytest.mark.parametrize("hq,hkv,t,n", MANY_ROWS)
@pytest.mark.parametrize("low", [((0, 128),), ((0, 400),), ((130, 384),), ((0, 129), (256, 650))])
@pytest.mark.parametrize("far", [False, True])
def test_many_rows_with_slots_of_no_weight(hq, hkv, t, n, low, far):
    """The first tiles of a range may have no weight at all, and the first logits after them any size."""
    _attend(hq, hkv, t, n, low=low, edit=_rest_far_below(low[-1][1]) if far else None, every=39)


@pytest.mark.parametrize("hq,hkv,t,n", [FEW_ROWS[1], FEW_ROWS[4]] + MANY_ROWS)
@pytest.mark.parametrize("lo,hi", [(0, 128), (140, 400)])
def test_slots_of_the_lowest_value(hq, hkv, t, n, lo, hi):
    """Logits of about -3e37, as far below the others as a float goes: no weight."""
    def edit(data):
        data["K"][0, :, lo:hi, 0] = 0xFF7F
    _attend(hq, hkv, t, n, edit=edit, every=39)


@pytest.mark.parametrize("hq,hkv,t,n", [FEW_ROWS[1], FEW_ROWS[4]] + MANY_ROWS[:3])
@pytest.mark.parametrize("value", [3e9, -3e9, -1e20, 1e30, -3.38e38])
def test_equal_logits_of_any_size(hq, hkv, t, n, value):
    """Every slot has the same logit, up to bf16's lowest value times the scale: equal weights."""
    def edit(data):
        data["K"][:] = 0
        data["K"][..., 0] = wl.f32_to_bf16_bits(np.float32([value]))[0]
    _attend(hq, hkv, t, n, edit=edit, every=39)


@pytest.mark.parametrize("hq,hkv,t", [(2, 2, 20), (64, 64, 40)])
def test_an_infinite_value_of_weight_zero(hq, hkv, t):
    """0 times infinity is NaN, whether the weight was lost inside a key range or between two."""
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    n = 640
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    q, K, V = (torch.randn(1, h, m, 128, generator=g, device="cuda").to(torch.bfloat16) for h, m in ((hq, t), (hkv, n), (hkv, n)))
    q[..., 0], K[..., 0], K[:, :, 0, 0] = 8.0, 0.0, 400.0   # slot 0 has a logit of 283, the others of about 0
    V[:, :, -1] = float("inf")
    counts = torch.ones(1, hkv, n, dtype=torch.int32, device="cuda")
    p = kb.make_params(K, V, hq, 8)
    ws = torch.empty(kb.kvs_workspace_size(p, n, t), dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(q)
    kb.kvs_decode_attn(p, q, K, V, counts, [n], out, ws)
    assert torch.isnan(out).all()


@pytest.mark.parametrize("hkv,first_round", [(2, 0), (90, 1)])
def test_window_rows_that_see_a_nan(hkv, first_round):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    n, W = 700, 24
    w = wl.small_case(seed=hkv, n_q_heads=hkv, n_kv_heads=hkv, window=W, seq_lens=(n,), budgets=(500,))
    data = wl.make_layer(w)
    data["K"][0, :, 300, 5] = NAN
    dev = tl.upload_layer(data)
    p = kb.make_params(dev["K"], dev["V"], hkv, W, first_round=first_round)
    ws = torch.empty(kb.kvs_workspace_size(p, n, 0), dtype=torch.uint8, device="cuda")
    o, lse = torch.zeros(1, hkv, W, 128, device="cuda"), torch.zeros(1, hkv, W, device="cuda")
    kb.kvs_window_stats(p, dev["K"], dev["V"], dev["counts"], dev["q_win"], [n], [500], ws, o_win=o, lse_win=lse)
    assert torch.isnan(o).all() and torch.isnan(lse).all()
