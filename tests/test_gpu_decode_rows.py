"""Decode attention of few query rows (at most 16 per KV head) at the edges of its blocks, column tiles and
clusters, against the oracle.

An output is the bf16 rounding of sum P' V / sum c P' with P' held in 16 significant bits: its error is at most
2^-17 max |V / c| < 1e-4 before the rounding, i.e. one bf16 ulp of the element where that is larger.  The
log-sum-exp carries the fp32 error of a logit (3e-6 of values below 20)."""
import numpy as np
import pytest

from oracle import kvs_oracle as oc
from paper_2603_00907_b200 import workloads as wl
from tests import kvs_testlib as tl

pytestmark = pytest.mark.gpu


# (query heads, KV heads, new tokens, lengths, token-major layout): 1, 4, 5, 8, 9 and 16 rows; lengths around the
# 16-slot block, one warp's, one CTA's and one cluster's share; long enough for several clusters per unit
@pytest.mark.parametrize("hq,hkv,t,lens,token_major", [
    (1, 1, 1, (1,), False), (4, 1, 1, (15, 16, 17), False), (5, 1, 1, (63, 64, 65, 129), True),
    (4, 2, 4, (511, 513, 200), False), (3, 1, 3, (2049, 0, 33), True), (8, 1, 1, (1025,), False),
    (4, 1, 1, (3500,), False), (2, 1, 7, (6200, 40), True), (16, 8, 1, tuple(range(17, 17 + 70)), False),
    # nine and sixteen rows on both sides of the lengths that go to the tensor-core tiles
    (9, 1, 1, (5632,), False), (9, 1, 1, (5633,), True), (4, 1, 4, (5700, 5650), False), (16, 1, 1, (16369,), False),
    # units for clusters of seven to one CTA in one wave of the GPU, and a ragged batch beyond it
    (36, 36, 1, (900,), False), (40, 20, 2, (800, 790), False), (50, 50, 3, (700,), False), (45, 45, 1, (600, 577), False),
    (24, 24, 1, (700, 640), True), (72, 24, 3, (333, 300, 301, 320, 310), False), (48, 48, 2, (90, 129, 128, 127), False),
    (40, 40, 1, (5200, 40, 33, 70), False)])
def test_decode_of_few_rows(hq, hkv, t, lens, token_major):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    B, n_max, G = len(lens), max(lens) + 3, hq // hkv
    w = wl.small_case(seed=hq + t, batch=B, n_q_heads=hq, n_kv_heads=hkv, window=8, seq_lens=(n_max,) * B,
                      budgets=(n_max,) * B, n_decode=t)
    data = wl.make_layer(w)
    rng = np.random.default_rng(3)
    data["counts"][:] = rng.integers(1, 9, size=data["counts"].shape)
    for b, n in enumerate(lens):                          # what lies behind a sequence must not matter
        data["K"][b, :, n:] = 0x7FC0
        data["V"][b, :, n:] = 0x7F80
        data["counts"][b, :, n:] = -7
    dev = tl.upload_layer(data)
    K, V = dev["K"], dev["V"]
    if token_major:
        K, V = (x.transpose(1, 2).contiguous().transpose(1, 2) for x in (K, V))
    p = kb.make_params(K, V, hq, 8)
    ws = torch.empty(kb.kvs_workspace_size(p, n_max, t), dtype=torch.uint8, device="cuda")
    out = torch.zeros((B, hq, t, 128), dtype=torch.bfloat16, device="cuda")
    lse = torch.zeros((B, hq, t), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    kb.kvs_decode_attn(p, dev["q_new"], K, V, dev["counts"], list(lens), out, ws, lse=lse, status_dev=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    og, lg = tl.bits_of(out), lse.cpu().numpy()
    for b, n in enumerate(lens):
        for h in range(hkv):
            hs = slice(h * G, (h + 1) * G)
            if n == 0:
                assert not og[b, hs].any() and not lg[b, hs].any()
                continue
            ref, lse_ref = oc.decode_attention(data["q_new"][b, hs], data["K"][b, h, :n], data["V"][b, h, :n],
                                               data["counts"][b, h, :n])
            ok, mx, _, _ = tl.bf16_close(og[b, hs], oc.f64_to_bf16(ref), atol=1e-4)
            assert ok, (b, h, mx)
            assert np.max(np.abs(lg[b, hs] - lse_ref)) < 1e-4


@pytest.mark.parametrize("hq,hkv,t,n", [(4, 1, 1, 40000), (16, 2, 2, 20011), (8, 2, 4, 9000)])
def test_stages_are_refilled_behind_their_use(hq, hkv, t, n):
    """Every warp fills its ring dozens of times: thirty passes over changing neighbours in the stream give the same bits,
    and those of the oracle's rounding for one head."""
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    w = wl.small_case(seed=n, n_q_heads=hq, n_kv_heads=hkv, window=8, seq_lens=(n,), budgets=(n,), n_decode=t)
    data = wl.make_layer(w)
    dev = tl.upload_layer(data)
    p = kb.make_params(dev["K"], dev["V"], hq, 8)
    ws = torch.empty(kb.kvs_workspace_size(p, n, t), dtype=torch.uint8, device="cuda")
    outs = []
    for _ in range(30):
        out = torch.zeros((1, hq, t, 128), dtype=torch.bfloat16, device="cuda")
        kb.kvs_decode_attn(p, dev["q_new"], dev["K"], dev["V"], dev["counts"], [n], out, ws)
        outs.append(out)
    assert all(torch.equal(o, outs[0]) for o in outs)
    G = hq // hkv
    ref, _ = oc.decode_attention(data["q_new"][0, :G], data["K"][0, 0], data["V"][0, 0], data["counts"][0, 0])
    ok, mx, _, _ = tl.bf16_close(tl.bits_of(outs[0])[0, :G], oc.f64_to_bf16(ref), atol=1e-4)
    assert ok, mx
