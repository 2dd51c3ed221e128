"""Time limits of a few microseconds, under which ordinary waits of the kernels run out at any point: behind the last request of
a CTA, with copies and tensor-core products in flight, in one role before the others.  Every call must return by itself,
with KVS_ERR_TIMEOUT or complete, and leave nothing behind that changes the next call."""
import pytest

pytestmark = pytest.mark.gpu

KVS_ERR_TIMEOUT = 6
LIMITS_US = (1, 2, 3, 5, 8, 15, 30)


@pytest.fixture(scope="module")
def kb():
    from paper_2603_00907_b200 import binding, build
    build.build()
    return binding


def _inputs(batch, hkv, n, rows, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    K, V, q = (torch.randn(batch, hkv, m, 128, generator=g, device="cuda").to(torch.bfloat16) for m in (n, n, rows))
    return K, V, torch.ones(batch, hkv, n, dtype=torch.int32, device="cuda"), q


def _outcomes(kb, call, clean, limits=LIMITS_US):
    """call() under every limit, each time followed by a call with the usual one that must repeat `clean`; the statuses."""
    import torch
    seen = set()
    for limit in limits:
        kb.kvs_debug_set_wait(limit, 0)
        try:
            status = call()[0]
            torch.cuda.synchronize()
        finally:
            kb.kvs_debug_set_wait(0, 0)
        seen.add(status.item())
        again = call()
        assert again[0].item() == 0
        for x, y in zip(again[1:], clean[1:]):
            assert torch.equal(x, y), limit
    assert seen <= {0, KVS_ERR_TIMEOUT}
    return seen


# (KV heads, sequences, slots, rows): one wave and several, ranges of many tiles, blocks of one and two steps, three query
# blocks, equal shares
@pytest.mark.parametrize("hkv,batch,n,rows", [(8, 1, 40000, 4), (160, 1, 9000, 4), (8, 2, 9000, 100), (4, 3, 5000, 300), (8, 24, 1300, 64)])
def test_statistics_leave_nothing_behind(kb, hkv, batch, n, rows):
    import torch
    K, V, counts, q = _inputs(batch, hkv, n, rows, n + rows)
    p = kb.make_params(K, V, hkv, rows, causal=False)
    ws = torch.empty(kb.kvs_workspace_size(p, n, 0), dtype=torch.uint8, device="cuda")

    def call():
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        out = [torch.zeros(batch, hkv, m, device="cuda") for m in (n, n, n // 2, n // 2)]
        kb.kvs_window_stats(p, K, V, counts, q, [n] * batch, [n // 2] * batch, ws, A=out[0], N1=out[1], score=out[2], w=out[3],
                            status_dev=status)
        return [status] + out

    clean = call()
    assert clean[0].item() == 0
    assert KVS_ERR_TIMEOUT in _outcomes(kb, call, clean)


@pytest.mark.parametrize("hkv,batch,n,rows", [(8, 1, 40000, 40), (64, 4, 3000, 128), (8, 1, 700, 20), (8, 8, 3000, 1), (8, 1, 9000, 16)])
def test_decode_leaves_nothing_behind(kb, hkv, batch, n, rows):
    import torch
    K, V, counts, q = _inputs(batch, hkv, n, rows, n + rows)
    p = kb.make_params(K, V, hkv, 32)
    ws = torch.empty(kb.kvs_workspace_size(p, n, rows), dtype=torch.uint8, device="cuda")

    def call():
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        out, lse = torch.zeros_like(q), torch.zeros(batch, hkv, rows, device="cuda")
        kb.kvs_decode_attn(p, q, K, V, counts, [n] * batch, out, ws, lse=lse, status_dev=status)
        return [status, out, lse]

    clean = call()
    assert clean[0].item() == 0
    _outcomes(kb, call, clean)


# KV heads, lengths, share of the pairs that merge: units of many tiles for all CTAs, for two CTAs each, for one CTA each
APART = [(8, [30000], 0.5), (8, [2600], 0.1), (8, [6000] * 16, 0.5), (8, [1200] * 36, 0.5)]
# units whose CTAs help one another (a CTA that gives up then holds tiles of several units)
HELPING = [(8, [4096] * 20, 0.3), (8, [28000, 12000, 18000, 3000, 600, 0, 20, 9000], 0.5)]


@pytest.mark.parametrize("hkv,lens,share", APART + HELPING)
@pytest.mark.parametrize("token_major", [False, True])
def test_a_compaction_stores_a_tile_whole_or_not_at_all(kb, hkv, lens, share, token_major):
    import torch
    batch, n_max, recent, off = len(lens), max(lens) + 3, 4, 32
    g = torch.Generator(device="cuda")
    g.manual_seed(batch + hkv)
    shape = (batch, n_max, hkv, 128) if token_major else (batch, hkv, n_max, 128)
    K0, V0 = (torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    if token_major:
        K0, V0 = K0.transpose(1, 2), V0.transpose(1, 2)
    counts0 = torch.randint(1, 1 << 20, (batch, hkv, n_max), generator=g, device="cuda", dtype=torch.int32)
    w = torch.rand(batch, hkv, n_max // 2, generator=g, device="cuda")
    mask = torch.zeros(batch, hkv, n_max // 2, dtype=torch.uint8, device="cuda")
    merged = []
    for b, n in enumerate(lens):
        pairs = max(0, (n - off - recent) // 2)
        merged.append(int(share * pairs))
        order = torch.rand(hkv, pairs, generator=g, device="cuda").argsort(-1)
        mask[b].scatter_(1, order[:, :merged[-1]], 1)
    p = kb.make_params(K0, V0, hkv, recent)
    ws = torch.empty(kb.kvs_workspace_size(p, n_max, 0), dtype=torch.uint8, device="cuda")
    index = torch.zeros(batch, hkv, n_max, dtype=torch.int32, device="cuda")

    def call(new_index=None):
        K, V, counts = (x.clone(memory_format=torch.preserve_format) for x in (K0, V0, counts0))
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        kb.kvs_compact(p, K, V, counts, mask, w, lens, merged, ws, new_index=new_index, status_dev=status)
        return [status, K, V, counts]

    clean = call(index)
    assert clean[0].item() == 0

    def rows(a, b):
        """[batch, heads, slots]: where key, value sum and count of the slot are the same in both caches."""
        return (a[1] == b[1]).all(-1) & (a[2] == b[2]).all(-1) & (a[3] == b[3])

    seen = set()
    moved = ~rows(clean, [None, K0, V0, counts0])          # slots that the compaction changes
    for limit in LIMITS_US:
        kb.kvs_debug_set_wait(limit, 0)
        try:
            got = call()
            torch.cuda.synchronize()
        finally:
            kb.kvs_debug_set_wait(0, 0)
        seen.add(got[0].item())
        done, still = rows(got, clean), rows(got, [None, K0, V0, counts0])
        for b, n in enumerate(lens):
            left = n - merged[b]
            # the tile that writes slot d is the one of the slots that move there
            tile = torch.zeros(hkv, left, dtype=torch.int64, device="cuda")
            if n <= off:
                continue
            src = torch.arange(n, device="cuda").expand(hkv, n)
            tile.scatter_(1, index[b, :, :n].long(), (src - off).clamp(min=0) // 64)
            ntiles = (n - off + 63) // 64
            m, d = moved[b, :, :left], done[b, :, :left]
            assert bool((d | still[b, :, :left]).all())
            stored, missing = (torch.zeros(hkv, ntiles, dtype=torch.int32, device="cuda").scatter_add_(1, tile, x.int())
                               for x in (m & d, m & ~d))
            assert not bool(((stored > 0) & (missing > 0)).any()), limit
            if got[0].item() == 0:
                assert int(missing.sum()) == 0
        again = call()
        assert again[0].item() == 0
        same = rows(again, clean)
        assert all(bool(same[b, :, :n - k].all()) for b, (n, k) in enumerate(zip(lens, merged)))
    assert KVS_ERR_TIMEOUT in seen and seen <= {0, KVS_ERR_TIMEOUT}
