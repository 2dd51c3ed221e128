"""The attention kernel's stabiliser is the maximum over a CTA's first tile of 128 slots.  Rows whose later logits
are larger by a little, by almost and by more than the range of an exponent of a part of the sum allows (2^60: the
CTA then walks its slots again with the true maxima), and rows whose first tiles are negligible, against the oracle.

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
