"""Attention launches that merge their own output rows, at the shapes where the split of a row decides
which code runs: rows spread over many thread blocks (one or few sequences), many rows inside one
block (short sequences), a row whose visual partials an earlier launch left, blocks of more layers
than one sweep feeds."""

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

# head_dim, heads, lengths (text, visual) per sequence
SHAPES = {
    "one_long_row_per_head": (128, 1, [(40, 2500)]),
    "rows_over_several_blocks": (64, 3, [(700, 900), (33, 1200)]),
    "many_rows_in_a_block": (128, 2, [(1 + i % 19, (7 * i) % 40) for i in range(23)]),
    "no_visual_tokens": (64, 4, [(15, 0), (16, 0), (17, 0)]),
}


def _dev(a, device):
    return torch.from_numpy(a.astype(np.int16)).view(torch.bfloat16).to(device).contiguous()


@pytest.mark.parametrize("mode", [qc.QC_MODE_VLA_QC, qc.QC_MODE_VLA_EQ8, qc.QC_MODE_GLA], ids=["qc", "eq8", "gla"])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_rows_merged_by_the_attention_launch(shape, mode):
    head_dim, heads, lens = SHAPES[shape]
    layer_kind = [0, 1, 1, 1, 1, 1, 0]   # a block of six layers (two sweeps), a layer alone
    n, b, steps = len(layer_kind), len(lens), 3
    longest = max(t + v for t, v in lens)
    w = W.Workload(95, "row_merge", n, heads, heads, head_dim, 16, b, 1, longest, longest, 1, steps, tuple(range(1, 6)))
    o = LazyAttentionOracle(n, heads, heads, head_dim, layer_kind, mode, n_seqs=b)
    sessions = [Session(n, heads, heads, head_dim, layer_kind, max_seqs=b, max_tokens_per_seq=longest + steps,
                        n_pages=2 * n * sum((t + steps + 31) // 16 + (v + 15) // 16 for t, v in lens), lazy_mode=mode,
                        poison_pool=True) for _ in range(2)]
    sessions[1].set_option("fused_merge", 0)
    for s in sessions:
        s.set_option("in_order_launches", 1)
    for i, (text, vis) in enumerate(lens):
        _, k, v = W.prefill_kv_np(w, i)
        k, v = k[:, :text + vis], v[:, :text + vis]
        kind = np.array([0] * text + [1] * vis, np.uint8)
        for s in sessions:
            s.prefill_append([i], [text + vis], kind, _dev(k, s.device), _dev(v, s.device))
        o.prefill_append(i, kind.tolist(), f64(k), f64(v))
    outs = [torch.empty((n, b, heads, head_dim), dtype=torch.bfloat16, device=s.device) for s in sessions]
    lses = [torch.empty((n, b, heads), dtype=torch.float32, device=s.device) for s in sessions]
    for step in range(steps):
        qn, kn, vn = W.decode_qkv_np(w, step)
        for s, out, lse in zip(sessions, outs, lses):
            s.decode_step(list(range(b)), _dev(qn, s.device), _dev(kn, s.device), _dev(vn, s.device), out, lse)
        for i in range(b):
            ref, ref_lse = o.decode_step(i, f64(qn[:, i]), f64(kn[:, i]), f64(vn[:, i]))
            for l in range(n):
                for out, lse in zip(outs, lses):
                    assert_close(bits_of(out)[l, i], ref[l], f"{shape} step {step} seq {i} layer {l}")
                    assert np.max(np.abs(lse.cpu().numpy()[l, i] - ref_lse[l])) <= 2e-3
    launches = [s.stats().kernel_launches for s in sessions]
    assert launches[0] < launches[1]   # the rows were merged without launches of their own
    for s in sessions:
        assert s.stats().device_error == 0
        s.close()


@pytest.mark.parametrize("row_cluster", [-1, 0], ids=["rows", "ranges"])
@pytest.mark.parametrize("shape", ["one_long_row_per_head", "rows_over_several_blocks"])
def test_the_same_step_gives_the_same_bits(shape, row_cluster):
    """Which block completes a row that several blocks share (tile ranges), and how many rows it completes, differs
    from run to run; the bits of the output may not."""
    head_dim, _, lens = SHAPES[shape]
    heads, b = 16, len(lens)
    layer_kind = [0, 1, 0, 1]
    n, longest = len(layer_kind), max(t + v for t, v in lens)
    s = Session(n, heads, heads, head_dim, layer_kind, max_seqs=b, max_tokens_per_seq=longest + 1,
                n_pages=2 * n * sum((t + 32) // 16 + (v + 15) // 16 for t, v in lens))
    s.set_option("in_order_launches", 1)
    s.set_option("row_cluster", row_cluster)
    gen = torch.Generator(device=s.device).manual_seed(3)

    def normal(*size):
        return torch.randn(size, generator=gen, device=s.device, dtype=torch.bfloat16)

    total = sum(t + v for t, v in lens)
    kind = np.concatenate([np.repeat(np.array([0, 1], np.uint8), (t, v)) for t, v in lens])
    k, v = normal(n, total, heads, head_dim), normal(n, total, heads, head_dim)
    qkv = [normal(n, b, heads, head_dim) for _ in range(3)]
    out, lse = torch.empty_like(qkv[0]), torch.empty((n, b, heads), dtype=torch.float32, device=s.device)
    first = None
    for run in range(60):
        s.prefill_append(list(range(b)), [t + v_ for t, v_ in lens], kind, k, v)
        launches = s.stats().kernel_launches
        s.decode_step(list(range(b)), *qkv, out, lse)
        assert s.stats().kernel_launches - launches == n + (1 if row_cluster else 2)   # set-up, with ranges their plan, a launch per layer
        got = (out.view(torch.int16).clone(), lse.view(torch.int32).clone())
        if first is None:
            first = got
        assert torch.equal(got[0], first[0]) and torch.equal(got[1], first[1]), f"run {run} differs from the first"
        for i in range(b):
            qc.qc_free_seq(s.cache, i)
    assert s.stats().device_error == 0
    s.close()


@pytest.mark.parametrize("options", [{}, {"in_order_launches": 1}, {"in_order_launches": 1, "row_cluster": 0},
                                     {"in_order_launches": 1, "fused_merge": 0}],
                         ids=["one_launch", "rows", "own_merge", "merge_launch"])
@pytest.mark.parametrize("q_heads,kv_heads", [(4, 4), (8, 2)])
def test_a_key_that_is_not_a_number_reaches_every_row_it_belongs_to(q_heads, kv_heads, options):
    """Softmax over a score that is not a number is not a number: a partial result that holds one may not be
    left out of the row, however many finite ones there are beside it."""
    n, b, text, vis, d, at, kv = 2, 2, 20, 700, 128, 333, 1
    s = Session(n, q_heads, kv_heads, d, [0, 1], max_seqs=b, max_tokens_per_seq=vis, n_pages=2 * n * b * 50)
    for key, value in options.items():
        s.set_option(key, value)
    gen = torch.Generator(device=s.device).manual_seed(5)

    def normal(*size):
        return torch.randn(size, generator=gen, device=s.device, dtype=torch.bfloat16)

    kind = np.array([0] * text + [1] * vis, np.uint8)
    k, v = normal(n, b * (text + vis), kv_heads, d), normal(n, b * (text + vis), kv_heads, d)
    k[0, text + at, kv, 7] = float("nan")   # the leader's, sequence 0, a visual token: its follower scores it too
    s.prefill_append([0, 1], [text + vis] * b, np.concatenate([kind] * b), k, v)
    q, kn, vn = normal(n, b, q_heads, d), normal(n, b, kv_heads, d), normal(n, b, kv_heads, d)
    out = torch.empty_like(q)
    s.decode_step([0, 1], q, kn, vn, out)
    group = q_heads // kv_heads
    hit = torch.zeros(n, b, q_heads, dtype=torch.bool, device=s.device)
    hit[:, 0, kv * group:(kv + 1) * group] = True
    assert torch.equal(torch.isnan(out).all(-1), hit) and torch.equal(torch.isnan(out).any(-1), hit)
    assert s.stats().device_error == 0
    s.close()


def test_a_shared_sweep_of_short_rows_is_not_slower_than_sweeps_of_its_own():
    """Many short sequences: what an item costs beyond its pages decides.  A GLA block moves fewer bytes than
    the same layers in VLA and has fewer sweeps; its leader's launch once took so much longer per item (its
    items alternated between two copies of the page loop) that the step was no faster."""
    n, b, heads, d, text, vis, steps = 10, 30, 16, 128, 110, 150, 8
    layer_kind = [1 if l >= 2 and (l - 2) % 4 else 0 for l in range(n)]
    best = {}
    for mode in (qc.QC_MODE_GLA, qc.QC_MODE_VLA_QC):
        s = Session(n, heads, heads, d, layer_kind, max_seqs=b, max_tokens_per_seq=vis + 100, n_pages=2 * n * b * 25, lazy_mode=mode)
        s.set_option("in_order_launches", 1)
        kind = np.tile(np.array([0] * text + [1] * vis, np.uint8), b)
        k, v = (torch.randn(n, len(kind), heads, d, device=s.device, dtype=torch.bfloat16) for _ in range(2))
        s.prefill_append(list(range(b)), [text + vis] * b, kind, k, v)
        q, kn, vn = (torch.randn(n, b, heads, d, device=s.device, dtype=torch.bfloat16) for _ in range(3))
        out = torch.empty_like(q)
        times = []
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(steps):
                s.decode_step(list(range(b)), q, kn, vn, out)
            e[1].record()
            torch.cuda.synchronize()
            times.append(e[0].elapsed_time(e[1]))
        best[mode] = min(times)
        s.close()
    assert best[qc.QC_MODE_GLA] < 0.9 * best[qc.QC_MODE_VLA_QC], best
