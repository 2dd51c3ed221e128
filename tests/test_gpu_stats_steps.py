"""Query blocks of every size class of the statistics kernel: up to 64 rows (one step per tile, the two accumulator
buffers in turn) and more (two steps of half the rows to a multiple of 16, so that the second ends in padding), with
one and with several query blocks, and three or more tiles per CTA.  Held to the tolerances of all statistics."""
import numpy as np
import pytest

from paper_2603_00907_b200 import workloads as wl
from tests import test_gpu_parity as parity

pytestmark = pytest.mark.gpu


# window rows per KV head: 1, 16, 24, 64 | 65, 80, 96, 126 | 130, 194, 224
@pytest.mark.parametrize("group,window", [(1, 1), (2, 8), (3, 8), (4, 16), (5, 13), (5, 16), (4, 24), (7, 18), (5, 26),
                                          (2, 97), (7, 32)])
def test_statistics_of_every_block_size(group, window):
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    hkv = 16
    w = wl.small_case(seed=100 + group * window, batch=1, n_q_heads=group * hkv, n_kv_heads=hkv, window=window,
                      seq_lens=(8000,), budgets=(7000,))
    data = wl.make_layer(w)
    parity._check_round_stats(kb, w, data["K"], data["V"], data["counts"], data["q_win"], list(w.seq_lens), group & 1)


@pytest.mark.parametrize("group,window,hkv", [(4, 16, 8), (5, 29, 4)])
def test_shares_that_cross_units(group, window, hkv):
    """192 units of up to five tiles, and 96 of two query blocks each: the kernel walks equal shares of all tiles, so
    most CTAs cross from one unit to the next, past a sequence that is done and past units of one ragged tile."""
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    lens = [1300, 1170, 400, 1290, 1301, 700, 1024, 300] * 3
    w = wl.small_case(seed=7, batch=len(lens), n_q_heads=group * hkv, n_kv_heads=hkv, window=window, seq_lens=tuple(lens),
                      budgets=tuple(n if i == 4 else n - n // 6 for i, n in enumerate(lens)))
    data = wl.make_layer(w)
    parity._check_round_stats(kb, w, data["K"], data["V"], data["counts"], data["q_win"], list(w.seq_lens), 1)


@pytest.mark.parametrize("mode", [1, 2])
def test_shares_that_cross_units_with_a_supplied_gradient(mode):
    """The same batch in the exact weight modes: two query operands instead of three are replaced from unit to unit.  Units
    at both ends of the walk and of a sequence, a short one, and one of two ragged tiles, against the oracle."""
    import torch
    from oracle import kvs_oracle as oc
    from paper_2603_00907_b200 import binding as kb, build
    from tests import kvs_testlib as tl
    build.build()
    lens = [1300, 1170, 400, 1290, 1301, 700, 1024, 300] * 3
    hkv, G, W = 8, 4, 16
    w = wl.small_case(seed=8, batch=len(lens), n_q_heads=G * hkv, n_kv_heads=hkv, window=W, seq_lens=tuple(lens),
                      budgets=tuple(n - n // 6 for n in lens))
    data = wl.make_layer(w)
    rng = np.random.default_rng(8)
    data["counts"][:] = rng.integers(1, 4, size=data["counts"].shape)
    E = wl.f32_to_bf16_bits(rng.standard_normal(data["q_win"].shape).astype(np.float32))
    dev, p, ws = parity._setup(kb, w, data)
    B, n_max = w.batch, w.n_max
    A, gs = (torch.zeros(B, hkv, n_max, device="cuda") for _ in range(2))
    gp = torch.zeros(B, hkv, n_max // 2, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    kb.kvs_window_stats_exact(p, dev["K"], dev["V"], dev["counts"], dev["q_win"], tl.to_dev_bf16(E), mode, lens,
                              list(w.budgets), ws, A=A, g_self=gs, g_pair=gp, status_dev=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    for b, h in ((0, 0), (0, 7), (1, 0), (2, 3), (7, 7), (11, 4), (15, 0), (23, 7)):
        n, hs = lens[b], slice(h * G, (h + 1) * G)
        st = oc.round_stats(data["K"][b, h, :n], data["V"][b, h, :n], data["counts"][b, h, :n].astype(np.int64),
                            data["q_win"][b, hs], w.budgets[b], 0, weight_mode=mode, E_bits=E[b, hs], **parity._oracle_kwargs(w))
        off, P, ab = st["off"], st["P"], st["Gabs"]
        ok, _, plain = tl.rel_close(A[b, h, off:off + 2 * P].cpu().numpy(), st["A"][off:off + 2 * P])
        assert ok, (b, h, plain)
        g = gs[b, h, off:off + 2 * P].cpu().numpy()
        for got, want, size in ((g[::2], st["G11"], ab[0]), (g[1::2], st["G22"], ab[1]), (gp[b, h, :P].cpu().numpy(), st["G12"], ab[2])):
            assert np.all(np.abs(got - want) <= tl.STAT_RTOL * size + 1e-37), (b, h)


@pytest.mark.parametrize("seed", [1, 2])
def test_values_around_a_mean(seed):
    """|vbar - o|^2 is a small difference of terms of about |mean|^2 = 128 here, and <vbar, o> comes from sixteen
    additions into an accumulator that is cut to 24 bits each time.  With the hi and lo terms of o in turn the partial
    sums grow evenly and the cuts add up to 8 * 2^-24 of the result, with all lo terms last to 12 * 2^-24: the error
    of N1 and N12 measured 0.96e-5 and 2.1e-5 of their norm in the first order, 1.4e-5 and 2.9e-5 in the second,
    in that proportion.  The bounds lie between."""
    import torch
    from oracle import kvs_oracle as oc
    from paper_2603_00907_b200 import binding as kb, build
    from tests import kvs_testlib as tl
    build.build()
    hq, hkv, n, W = 32, 8, 1024, 32
    w = wl.small_case(seed=60 + seed, n_q_heads=hq, n_kv_heads=hkv, window=W, seq_lens=(n,), budgets=(340,))
    data = wl.make_layer(w)
    rng = np.random.default_rng(seed)
    c = 1 + rng.exponential(12.0, size=(1, hkv, n)).astype(np.int32)
    mean = rng.standard_normal((1, hkv, 1, 128))
    values = rng.standard_normal((1, hkv, n, 128)) * np.sqrt(c)[..., None] + mean * c[..., None]
    data["counts"][:], data["V"] = c, wl.f32_to_bf16_bits(values.astype(np.float32))
    dev = tl.upload_layer(data)
    p = kb.make_params(dev["K"], dev["V"], hq, W)
    ws = torch.empty(kb.kvs_workspace_size(p, n, 0), dtype=torch.uint8, device="cuda")
    N1, N12 = torch.zeros(1, hkv, n, device="cuda"), torch.zeros(1, hkv, n // 2, device="cuda")
    kb.kvs_window_stats(p, dev["K"], dev["V"], dev["counts"], dev["q_win"], [n], [340], ws, N1=N1, N12=N12)
    err, ref = np.zeros(2), np.zeros(2)
    for h in range(hkv):
        st = oc.round_stats(data["K"][0, h], data["V"][0, h], c[0, h], data["q_win"][0, 4 * h:4 * h + 4], 340, 0,
                            **parity._oracle_kwargs(w))
        off, P = st["off"], st["P"]
        for i, (got, want) in enumerate(((N1[0, h, off:off + 2 * P], st["N1"][off:off + 2 * P]),
                                         (N12[0, h, :P], st["N12"][:P]))):
            err[i] += np.sum((got.cpu().numpy() - want) ** 2)
            ref[i] += np.sum(want ** 2)
    rel = np.sqrt(err / ref)
    assert rel[0] < 1.15e-5 and rel[1] < 2.4e-5, rel


@pytest.mark.parametrize("scale", [3e-18, 2e-20, 0.0])
def test_cosine_of_short_keys(scale):
    """Every second key is `scale` times as long: the cosine with its neighbour does not depend on it until the product
    of the lengths is below 1e-30, where it is 0 (in float64 as in float32)."""
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    w = wl.small_case(seed=77, window=8, seq_lens=(700,), budgets=(500,))
    data = wl.make_layer(w)
    keys = (data["K"].astype(np.uint32) << 16).view(np.float32)
    keys[:, :, ::2] *= np.float32(scale)
    data["K"] = wl.f32_to_bf16_bits(keys)
    parity._check_round_stats(kb, w, data["K"], data["V"], data["counts"], data["q_win"], [700], 0)
