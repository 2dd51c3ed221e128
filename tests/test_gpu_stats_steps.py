"""Query blocks of every size class of the statistics kernel: up to 64 rows (one step per tile, the two accumulator
buffers in turn) and more (two steps of half the rows to a multiple of 16, so that the second ends in padding), with
one and with several query blocks, and three or more tiles per CTA.  Held to the tolerances of all statistics."""
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
