"""How the launches of a step are cut is chosen from the numbers of rows and pages: a choice that is slower than
the library's other way of cutting the same step is a wrong choice.  Sizes where the places for thread blocks run
out, or where a few rows are most of the work."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2602_01901_b200 import binding as qc
from paper_2602_01901_b200.session import Session

pytestmark = pytest.mark.gpu


def _us_per_layer(s, n, b, steps=16):
    """Best of three runs of `steps` steps, microseconds per layer."""
    q = torch.randn(n, b, s.hq, s.d, device=s.device, dtype=torch.bfloat16)
    k = torch.randn(n, b, s.hkv, s.d, device=s.device, dtype=torch.bfloat16)
    out, ids, best = torch.empty_like(q), list(range(b)), float("inf")
    for _ in range(3):
        for _ in range(3):
            s.decode_step(ids, q, k, k, out)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        torch.cuda._sleep(3_000_000)   # the steps queue up behind this
        e[0].record()
        for _ in range(steps):
            s.decode_step(ids, q, k, k, out)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) * 1e3 / steps / n)
    return best


def _not_slower_than_ranges(hq, hkv, d, layer_kind, mode, lens, margin=1.12, other=("row_cluster", 0)):
    n, b = len(layer_kind), len(lens)
    s = Session(n, hq, hkv, d, layer_kind, max_seqs=b, max_tokens_per_seq=max(map(max, lens)) + 512,
                n_pages=2 * n * sum(t // 16 + v // 16 + 34 for t, v in lens), lazy_mode=mode)
    s.set_option("in_order_launches", 1)
    for i, (text, vis) in enumerate(lens):
        k = torch.randn(n, text + vis, hkv, d, device=s.device, dtype=torch.bfloat16)
        s.prefill_append([i], [text + vis], np.array([0] * text + [1] * vis, np.uint8), k, k)
    as_it_comes = (other[0], {"row_cluster": -1, "row_warps": 0}[other[0]])
    chosen = us = float("inf")
    for _ in range(4):   # (a host that stalls while the steps queue up makes either slower: the best of a few tries)
        s.set_option(*as_it_comes)
        chosen = min(chosen, _us_per_layer(s, n, b))
        s.set_option(*other)
        us = min(us, _us_per_layer(s, n, b))
        if chosen <= margin * us:
            break
    assert s.stats().device_error == 0
    s.close()
    assert chosen <= margin * us, f"as chosen {chosen:.1f} us a layer, with {other[0]} {other[1]} {us:.1f}"


BLOCKS_OF_4, BLOCKS_OF_2 = [0, 1, 1, 1] * 2, [0, 1] * 2


@pytest.mark.parametrize("hq,hkv,block,mode,batch,tokens", [
    (28, 4, BLOCKS_OF_4, qc.QC_MODE_GLA, 4, 1000),     # 16 rows: clusters of eight are resident fifteen times
    (28, 4, BLOCKS_OF_4, qc.QC_MODE_VLA_QC, 20, 1000),   # 80 rows, one thread block per SM
    (32, 8, BLOCKS_OF_4, qc.QC_MODE_GLA, 20, 1000),    # 160 rows, more than places
    (28, 4, BLOCKS_OF_2, qc.QC_MODE_VLA_QC, 18, 3000),   # 72 rows: clusters of four are resident 71 times
    (34, 34, BLOCKS_OF_2, qc.QC_MODE_VLA_QC, 1, 8000),   # 34 rows: clusters of eight are resident 33 times
    (40, 40, BLOCKS_OF_2, qc.QC_MODE_VLA_QC, 32, 300),   # 1 280 rows of one warp: an SM holds eight clusters at most
])
def test_rows_get_no_more_thread_blocks_than_are_resident(hq, hkv, block, mode, batch, tokens):
    _not_slower_than_ranges(hq, hkv, 128, block, mode, [(60, tokens - 60)] * batch)


@pytest.mark.parametrize("heads,d,lens,warps", [
    (30, 64, [(60, 940)] * 30, 2),                                            # 900 rows: an SM holds eight blocks of two warps
    (40, 128, [(20 + i % 30, 5 + 7 * i % 41) for i in range(32)], 1),         # 1 280 uneven rows: blocks of three warps in a third wave
], ids=["64_wide", "uneven"])
def test_rows_of_many_sequences_get_the_warps_that_are_resident(heads, d, lens, warps):
    _not_slower_than_ranges(heads, heads, d, BLOCKS_OF_2, qc.QC_MODE_VLA_QC, lens, other=("row_warps", warps))


@pytest.mark.parametrize("heads,d,batch,tokens,block,mode", [
    (40, 64, 1, 10400, BLOCKS_OF_2, qc.QC_MODE_VLA_EQ8),    # clusters of four on 160 of 296 places
    (32, 64, 3, 3140, [0, 0, 0, 0], qc.QC_MODE_VLA_QC),     # of two on 192
    (16, 64, 1, 9700, [0, 0, 0, 0], qc.QC_MODE_VLA_QC),     # of eight on 128
    (4, 64, 10, 5060, [0, 0, 0, 0], qc.QC_MODE_VLA_QC),     # of four on 160
    (32, 64, 10, 2130, [0, 0, 0, 0], qc.QC_MODE_VLA_QC),    # 320 blocks of four warps on 592 places
    (40, 128, 32, 1240, BLOCKS_OF_4, qc.QC_MODE_VLA_EQ8),   # a warp for each of 1 280 rows
])
def test_long_rows_on_part_of_the_chip(heads, d, batch, tokens, block, mode):
    _not_slower_than_ranges(heads, heads, d, block, mode, [(100, tokens - 100)] * batch, margin=1.05)


@pytest.mark.parametrize("heads,d,tokens", [(8, 128, 32000), (4, 64, 32000), (2, 128, 48000)])
def test_a_few_very_long_rows_use_the_whole_chip(heads, d, tokens):
    _not_slower_than_ranges(heads, heads, d, BLOCKS_OF_2, qc.QC_MODE_VLA_QC, [(100, tokens)])


@pytest.mark.parametrize("heads,d,lens", [
    (16, 128, [(18, 4000), (4000, 18)] * 7),
    (16, 64, [(60, int(7900 * f)) for f in (1, .62, .75, .68, .97, .88, .71, .82)]),
    (16, 128, [(60, int(3900 * (1 - 0.035 * i))) for i in range(15)]),
], ids=["text_of_half_the_batch", "64_wide", "six_tenths_to_one"])
def test_rows_that_are_longer_than_others_by_many_pages(heads, d, lens):
    _not_slower_than_ranges(heads, heads, d, BLOCKS_OF_2, qc.QC_MODE_VLA_QC, lens, margin=1.05)


@pytest.mark.parametrize("hq,hkv,d,lens", [
    (32, 32, 128, [(3000, 16)] + [(16, 3000)] * 7),
    (32, 8, 64, [(26, 8800), (8800, 26)] * 2 + [(26, 8800)]),
    (40, 40, 128, [(56, 1839), (1839, 56)] * 7 + [(56, 1839)]),
])
def test_a_follower_whose_text_is_mostly_one_sequences_is_not_slower_than_ranges(hq, hkv, d, lens):
    _not_slower_than_ranges(hq, hkv, d, BLOCKS_OF_2, qc.QC_MODE_VLA_QC, lens)


@pytest.mark.parametrize("hq,hkv", [(4, 4), (8, 2)])
@pytest.mark.parametrize("key,value", [("static_min_tiles", 7), ("static_row_cost", 9), ("static_partition", 1), ("plan_ahead", 0),
                                       ("fused_merge", 0), ("fold_append", 0), ("row_cluster", 0)])
def test_an_option_of_the_tile_ranges_is_answered_by_tile_ranges(key, value, hq, hkv):
    n, b = 4, 2
    s = Session(n, hq, hkv, 128, [0, 1, 0, 1], max_seqs=b, max_tokens_per_seq=400, n_pages=2 * n * b * 30)
    s.set_option("in_order_launches", 1)
    k = torch.randn(n, 330 * b, hkv, 128, device=s.device, dtype=torch.bfloat16)
    s.prefill_append([0, 1], [330] * b, np.array(([0] * 30 + [1] * 300) * b, np.uint8), k, k)
    q, out = (torch.randn(n, b, hq, 128, device=s.device, dtype=torch.bfloat16) for _ in range(2))
    new = torch.randn(n, b, hkv, 128, device=s.device, dtype=torch.bfloat16)

    def launches():
        before = s.stats().kernel_launches
        s.decode_step([0, 1], q, new, new, out)
        return s.stats().kernel_launches - before

    assert launches() == 1 + n     # set-up, and a launch that finishes its rows for each layer
    s.set_option(key, value)
    assert launches() > 1 + n      # a plan, an append or merges besides
    assert s.stats().device_error == 0
    s.close()
