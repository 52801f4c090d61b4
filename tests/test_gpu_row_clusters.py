"""Attention launches that give every output row a cluster of thread blocks, against the oracle, at the
shapes where the dealing of a row's pages over a cluster's warps can go wrong: fewer pages than warps,
pages that fill up during the steps, no visual tokens, more pages of a warp than its page-id list
holds, every number of followers, query groups of one and two slices."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle.lazy_attention import LazyAttentionOracle
from paper_2602_01901_b200 import binding as qc
from paper_2602_01901_b200 import workloads as W
from paper_2602_01901_b200.session import Session, bits_of
from parity_util import assert_close, f64

pytestmark = pytest.mark.gpu

# head_dim, query heads, KV heads, followers per leader, lengths (text, visual) per sequence, CTAs per row (of six
# warps) or warps of a row's only CTA
SHAPES = {
    "a_page_or_two": (128, 2, 2, 1, [(1, 0), (14, 3), (15, 1), (16, 16)], 8),
    "fewer_pages_than_warps": (64, 3, 3, 2, [(30, 65), (47, 0), (33, 17)], 4),
    "three_followers": (128, 2, 2, 3, [(95, 700), (31, 512)], 3),
    "long_page_lists": (128, 1, 1, 1, [(40, 3300)], 1),
    "group_of_seven": (128, 14, 2, 1, [(31, 300), (15, 129), (64, 0)], 2),
    "group_three_followers": (128, 4, 1, 3, [(47, 500)], 8),
    "group_in_two_slices": (64, 24, 2, 2, [(33, 250), (16, 90)], 5),
    "four_warps": (128, 2, 2, 1, [(30, 200), (47, 190)], "row_warps 4"),
    "three_warps": (64, 3, 3, 2, [(33, 17), (16, 95)], "row_warps 3"),
    "two_warps": (128, 2, 2, 3, [(15, 300), (1, 0)], "row_warps 2"),
    "one_warp": (128, 2, 2, 1, [(47, 700), (14, 33)], "row_warps 1"),
    "as_chosen": (128, 8, 2, 1, [(35, 400), (50, 380)], -1),
}


def _dev(a, device):
    return torch.from_numpy(a.astype(np.int16)).view(torch.bfloat16).to(device).contiguous()


@pytest.mark.parametrize("mode", [qc.QC_MODE_VLA_QC, qc.QC_MODE_VLA_EQ8, qc.QC_MODE_GLA], ids=["qc", "eq8", "gla"])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_a_cluster_per_row(shape, mode):
    head_dim, hq, hkv, followers, lens, cluster = SHAPES[shape]
    layer_kind = [0] + [0] + [1] * followers + [0, 1]
    n, b, steps = len(layer_kind), len(lens), 3
    longest = max(t + v for t, v in lens)
    w = W.Workload(96, "row_clusters", n, hq, hkv, head_dim, 16, b, 1, longest, longest, 1, steps,
                   tuple(l for l in range(n) if layer_kind[l]))
    o = LazyAttentionOracle(n, hq, hkv, head_dim, layer_kind, mode, n_seqs=b)
    s = Session(n, hq, hkv, head_dim, layer_kind, max_seqs=b + 1, max_tokens_per_seq=longest + steps,
                n_pages=2 * n * sum((t + steps + 31) // 16 + (v + 15) // 16 for t, v in lens), lazy_mode=mode, poison_pool=True)
    s.set_option("in_order_launches", 1)
    option, value = cluster.split() if isinstance(cluster, str) else ("row_cluster", cluster)
    s.set_option(option, int(value))
    ids = list(range(b, 0, -1))
    for i, (text, vis) in enumerate(lens):
        _, k, v = W.prefill_kv_np(w, i)
        k, v = k[:, :text + vis], v[:, :text + vis]
        kind = np.array([0] * text + [1] * vis, np.uint8)
        s.prefill_append([ids[i]], [text + vis], kind, _dev(k, s.device), _dev(v, s.device))
        o.prefill_append(i, kind.tolist(), f64(k), f64(v))
    out = torch.empty((n, b, hq, head_dim), dtype=torch.bfloat16, device=s.device)
    lse = torch.empty((n, b, hq), dtype=torch.float32, device=s.device)
    leader = [max(x for x in range(l + 1) if not layer_kind[x]) for l in range(n)]
    for step in range(steps):
        launches = s.stats().kernel_launches
        qn, kn, vn = W.decode_qkv_np(w, step)
        s.decode_step(ids, _dev(qn, s.device), _dev(kn, s.device), _dev(vn, s.device), out, lse)
        for i in range(b):
            ref, ref_lse = o.decode_step(i, f64(qn[:, i]), f64(kn[:, i]), f64(vn[:, i]))
            for l in range(n):
                assert_close(bits_of(out)[l, i], ref[l], f"{shape} step {step} seq {i} layer {l}")
                assert np.max(np.abs(lse.cpu().numpy()[l, i] - ref_lse[l])) <= 2e-3
        assert s.stats().kernel_launches - launches == 1 + n   # set-up, and one launch for each layer
    # the new rows and the Q Cache, bit for bit
    for i, sid in enumerate(ids):
        _, n_text, _ = s.page_table(0, qc.QC_STREAM_V_TEXT, sid)
        for l in range(n):
            owner = leader[l] if mode == qc.QC_MODE_GLA else l
            for h in range(hkv):
                assert np.array_equal(s.read_row(l, qc.QC_STREAM_V_TEXT, sid, n_text - 1, h), vn[l, i, h])
                assert np.array_equal(s.read_row(l, qc.QC_STREAM_K_TEXT, sid, n_text - 1, h), kn[owner, i, h])
            assert np.array_equal(s.read_qcache(l)[sid], qn[leader[l], i])
    assert s.stats().device_error == 0
    s.close()


@pytest.mark.parametrize("entry", ["step", "layers"])
@pytest.mark.parametrize("options", [{}, {"row_cluster": 0}, {"plan_ahead": 0}], ids=["rows", "ranges", "unplanned_ranges"])
@pytest.mark.parametrize("hq,hkv", [(4, 4), (8, 2)])
def test_steps_enqueued_without_a_wait_between_them(hq, hkv, options, entry):
    """The first launch of a step comes right after the one that writes the step's descriptors and new page-table
    entries, in a stack of two layers every second one does: sequences in another order each step, pages that fill up
    every few steps, nothing that lets one step finish before the next is enqueued."""
    n, d, b, steps = 2, 128, 4, 48
    text, vis = [29, 33, 38, 44], [200, 190, 180, 170]
    s = Session(n, hq, hkv, d, [0, 0], max_seqs=b, max_tokens_per_seq=256, n_pages=2 * n * b * 24, poison_pool=True)
    for key, value in {"in_order_launches": 1, **options}.items():
        s.set_option(key, value)
    o = LazyAttentionOracle(n, hq, hkv, d, [0, 0], qc.QC_MODE_VLA_QC, n_seqs=b)
    gen = torch.Generator().manual_seed(21)

    def normal(*size):
        return torch.randn(size, generator=gen).to(torch.bfloat16)

    for i in range(b):
        kind = np.array([0] * text[i] + [1] * vis[i], np.uint8)
        k, v = normal(n, len(kind), hkv, d), normal(n, len(kind), hkv, d)
        s.prefill_append([i], [len(kind)], kind, k.to(s.device), v.to(s.device))
        o.prefill_append(i, kind.tolist(), k.double().numpy(), v.double().numpy())
    q, k, v = normal(steps, n, b, hq, d), normal(steps, n, b, hkv, d), normal(steps, n, b, hkv, d)
    orders = [torch.randperm(b, generator=gen).tolist() for _ in range(steps)]
    dq, dk, dv = (t.to(s.device) for t in (q, k, v))
    out = torch.empty_like(dq)
    launches = s.stats().kernel_launches
    torch.cuda._sleep(20_000_000)   # the steps queue up behind this
    for i in range(steps):
        if entry == "step":
            s.decode_step(orders[i], dq[i], dk[i], dv[i], out[i])
        else:
            s.decode_begin(orders[i])
            for l in range(n):
                s.decode_layer(l, dq[i, l], dk[i, l], dv[i, l], out[i, l])
    assert s.stats().device_error == 0
    # set-up, the plan of tile ranges, a launch per layer and the merge launches that these leave
    merges = 0 if not options or (hq == hkv and "plan_ahead" not in options) else n
    assert s.stats().kernel_launches - launches == (1 + ("row_cluster" in options) + n + merges) * steps
    got = bits_of(out)
    for i in range(steps):
        for at, seq in enumerate(orders[i]):
            ref, _ = o.decode_step(seq, *(t[i, :, at].double().numpy() for t in (q, k, v)))
            for l in range(n):
                assert_close(got[i, l, at], ref[l], f"step {i} sequence {seq} layer {l}")
    s.close()
