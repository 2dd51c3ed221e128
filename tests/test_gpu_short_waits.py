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
