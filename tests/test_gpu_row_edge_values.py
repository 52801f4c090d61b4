"""Values that arithmetic has to be careful with, in launches that give every output row thread blocks of
its own: infinite value elements, keys whose scores are minus infinity, pieces of a row whose weight underflows.
The oracle's definition decides: a key of weight zero counts for nothing, an infinite value of a key that
counts makes its element of the row infinite and leaves the others alone."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle.lazy_attention import LazyAttentionOracle
from paper_2602_01901_b200 import binding as qc
from paper_2602_01901_b200.session import Session, bits_of
from parity_util import assert_close, f64

pytestmark = pytest.mark.gpu

HEADS = [(2, 2, 128), (8, 2, 128), (3, 3, 64)]   # query heads, KV heads, head_dim


def _case(split, heads, mode, visual, change):
    """Two layers (a leader and its follower), one sequence of 16 text and `visual` visual tokens; `change` edits
    q, k, v and returns what the oracle is given in place of k and v.  Returns outputs and the oracle's."""
    hq, hkv, d = heads
    text, n = 16, 2
    gen = torch.Generator().manual_seed(11)

    def normal(*size):
        return torch.randn(size, generator=gen, dtype=torch.float32).to(torch.bfloat16)

    q, kn, vn = normal(n, 1, hq, d), normal(n, 1, hkv, d), normal(n, 1, hkv, d)
    k, v = normal(n, text + visual, hkv, d), normal(n, text + visual, hkv, d)
    q = q.abs() + 0.25   # every query element positive: a key's sign decides its score's
    ok, ov = change(k, v, text)
    s = Session(n, hq, hkv, d, [0, 1], max_tokens_per_seq=text + visual + 1, n_pages=2 * n * (visual // 16 + 4), lazy_mode=mode)
    s.set_option("in_order_launches", 1)
    s.set_option(*split)
    o = LazyAttentionOracle(n, hq, hkv, d, [0, 1], mode, n_seqs=1)
    kind = np.array([0] * text + [1] * visual, np.uint8)
    s.prefill_append([0], [text + visual], kind, k.to(s.device), v.to(s.device))
    out = torch.empty((n, 1, hq, d), dtype=torch.bfloat16, device=s.device)
    before = s.stats().kernel_launches
    s.decode_step([0], q.to(s.device), kn.to(s.device), vn.to(s.device), out)
    assert s.stats().kernel_launches - before == 1 + n   # set-up, and a launch that finishes its rows for each layer
    assert s.stats().device_error == 0
    o.prefill_append(0, kind.tolist(), ok.double().numpy(), ov.double().numpy())
    ref, _ = o.decode_step(0, q[:, 0].double().numpy(), kn[:, 0].double().numpy(), vn[:, 0].double().numpy())
    got = f64(bits_of(out))[:, 0]
    s.close()
    return got, np.asarray(ref)


def _cases(splits):
    return [pytest.param(split, heads, mode, id=f"{split[0]}_{split[1]}-{heads[0]}_{heads[1]}_{heads[2]}-{name}")
            for split in splits for heads in HEADS if split[0] == "row_cluster" or heads[0] == heads[1]
            for mode, name in ((qc.QC_MODE_VLA_QC, "qc"), (qc.QC_MODE_GLA, "gla"))]


# (splits that give the page a warp of its own)
@pytest.mark.parametrize("split,heads,mode", _cases([("row_cluster", 1), ("row_cluster", 3), ("row_cluster", 8), ("row_warps", 4)]))
def test_a_page_without_weight_counts_for_nothing(split, heads, mode):
    def change(k, v, text):
        at = slice(text + 32, text + 48)            # the third visual page: scores some 1 000 below the others'
        k[:, at] = -60.0
        ov = v.clone()
        v[:, text + 35, :, 5] = float("inf")
        return k, ov

    got, ref = _case(split, heads, mode, 64, change)
    assert np.isfinite(got).all()
    assert_close(torch.from_numpy(got).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16), ref, "page without weight")


def _check_infinite(got, ref):
    """Infinite elements where the oracle has them, with its signs, and the others as close as ever."""
    hit = np.isinf(ref)
    assert hit.any() and np.array_equal(got[hit], ref[hit])
    rest, ref_rest = np.where(hit, 0.0, got), np.where(hit, 0.0, ref)
    assert_close(torch.from_numpy(rest).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16), ref_rest, "finite elements")


@pytest.mark.parametrize("split,heads,mode", _cases([("row_cluster", 3), ("row_cluster", 5), ("row_warps", 2)]))
def test_an_infinite_value_makes_its_element_infinite_and_no_other(split, heads, mode):
    def change(k, v, text):
        # pages 13 and 25 of the 40: with three, resp. five thread blocks per row they are the last one's
        v[:, text + 13 * 16 + 7, :, 5] = float("inf")
        v[:, text + 25 * 16, :, 9] = -float("inf")
        return k, v

    _check_infinite(*_case(split, heads, mode, 640, change))


@pytest.mark.parametrize("split,heads,mode", _cases([("row_cluster", 1), ("row_cluster", 2), ("row_cluster", 8), ("row_warps", 1),
                                                     ("row_warps", 3)]))
def test_pages_of_keys_that_score_minus_infinity_count_for_nothing(split, heads, mode):
    def change(k, v, text):
        # all of the prompt's text and the second and third of 12 visual pages: the first page that some warp meets
        k[:, :text, :, 0] = -float("inf")
        k[:, text + 16:text + 48, :, 0] = -float("inf")
        return k, v

    got, ref = _case(split, heads, mode, 192, change)
    assert np.isfinite(got).all()
    assert_close(torch.from_numpy(got).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16), ref, "masked pages")
