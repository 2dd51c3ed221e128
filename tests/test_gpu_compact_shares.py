"""Compaction of batches whose units differ in length: CTAs that are done with their own unit go on with others.  Every
sequence must come out as it does in a call of its own, where there is no other unit of another length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# KV heads, slots of every sequence (0 and lengths inside the protected prefix among them), share of the pairs that merge
@pytest.mark.parametrize("hkv,lens,share", [
    (8, [20011, 600, 4099, 0, 20, 9000, 1200, 700], 0.5), (1, [70001] + [2100 + 13 * i for i in range(40)], 0.9),
    (4, [300] * 60 + [30000], 0.02), (8, [6400] * 37, 0.5), (2, [33, 34, 36000, 65, 66, 129], 0.4)])
@pytest.mark.parametrize("token_major", [False, True])
def test_units_of_different_lengths(hkv, lens, share, token_major):
    import torch
    from paper_2603_00907_b200 import binding as kb, build
    build.build()
    rng = np.random.default_rng(len(lens) + hkv)
    g = torch.Generator(device="cuda")
    g.manual_seed(hkv)
    batch, n_max, recent = len(lens), max(lens) + 5, 4
    shape = (batch, n_max, hkv, 128) if token_major else (batch, hkv, n_max, 128)
    K, V = (torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    if token_major:
        K, V = K.transpose(1, 2), V.transpose(1, 2)
    counts = torch.randint(1, 50, (batch, hkv, n_max), generator=g, device="cuda", dtype=torch.int32)
    w = torch.rand(batch, hkv, n_max // 2, generator=g, device="cuda")
    pairs = [max(0, (n - 32 - recent) // 2) for n in lens]
    merged = [int(share * p) for p in pairs]
    mask = np.zeros((batch, hkv, n_max // 2), np.uint8)
    for b in range(batch):
        for h in range(hkv):
            mask[b, h, rng.permutation(pairs[b])[:merged[b]]] = 1
    mask = torch.from_numpy(mask).cuda()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def compact(rows):
        k, v, c = (x[rows].clone(memory_format=torch.preserve_format) for x in (K, V, counts))
        p = kb.make_params(k, v, hkv, recent)
        ws = torch.empty(kb.kvs_workspace_size(p, n_max, 0), dtype=torch.uint8, device="cuda")
        index = torch.full((len(rows), hkv, n_max), -1, dtype=torch.int32, device="cuda")
        m = [merged[b] for b in rows]
        new = kb.kvs_compact(p, k, v, c, mask[rows], w[rows], [lens[b] for b in rows], m, ws, new_index=index, status_dev=status)
        assert new == [lens[b] - merged[b] for b in rows]
        return k, v, c, index

    got = compact(list(range(batch)))
    for b in range(batch):
        n, left = lens[b], lens[b] - merged[b]
        for x, y, m in zip(got, compact([b]), (left, left, left, n)):
            x, y = x[b][:, :m], y[0][:, :m]
            assert torch.equal(x if x.dtype == torch.int32 else x.view(torch.int16), y if y.dtype == torch.int32 else y.view(torch.int16))
    assert status.item() == 0


# Sizes at which the CTAs do help one another, and one that a shared launch leaves to itself for its short units.
HELPED = [(8, [28000, 12000, 18000, 3000, 600, 0, 20, 9000], 0.5), (8, [4096] * 20, 0.9), (8, [8000, 5000, 7600, 4300] * 8, 0.02),
          (8, [6000, 7500, 4800] * 6, 0.4)]
NOT_HELPED = [(8, [1120] * 24, 0.5)]


@pytest.mark.parametrize("hkv,lens,share", HELPED + NOT_HELPED)
@pytest.mark.parametrize("token_major", [False, True])
def test_units_that_are_helped(hkv, lens, share, token_major):
    test_units_of_different_lengths(hkv, lens, share, token_major)
