"""What a program that serves a multimodal model has this library do, as cases to time.

One pass is the life of a batch of sequences: their prompts enter the cache, tokens are generated,
the sequences are released.  (A decode step makes its sequences longer and nothing makes them shorter
again, so a pass that can be repeated on one cache has to begin with the prompts and end with the
release; it is also what a serving process does.)  The prompts' K/V are stored by qc_prefill_append
(``attend`` false: they were computed elsewhere, as on a decode node) or attended and stored by
qc_prefill_attend, in ``chunks`` calls; a case with two turns attends a second, text-only prompt on
top of what the sequences hold and generates again.  ``entry`` is how a step is issued:

    layers     qc_decode_begin and one qc_decode_layer per layer, as a model calls it that has a
               layer's q/k/v only after the layer before it has run
    in_order   qc_decode_step under the schedule with one launch per layer (what bench.py reports)
    step       qc_decode_step as it comes: every layer's q/k/v are there when the step begins
    host       qc_decode_step_host on pinned host buffers

Shapes are those of ``workloads.py`` (the five benchmark shapes and the one with 22 of 32 layers
lazy) with fewer generated tokens, or smaller ones of the same kind.  Values are N(0, 1) in bf16, as
everywhere in this repository: rotated and normalised queries and keys are close to that, and the
scores then are N(0, 1) after the softmax scale.  Lengths differ between the sequences of a batch
where ``ragged`` is set.
"""

from __future__ import annotations

import numpy as np
import torch

from paper_2602_01901_b200 import binding as qc
from paper_2602_01901_b200.session import Session

MODES = {"vla_qc": qc.QC_MODE_VLA_QC, "vla_eq8": qc.QC_MODE_VLA_EQ8, "gla": qc.QC_MODE_GLA}


def _case(name, **fields):
    case = dict(layers=32, q_heads=32, kv_heads=32, head_dim=128, paged=True, batch=1, text_before=35, visual=576,
                text_after=64, ragged=False, lazy="every_second", mode="vla_qc", attend=False, chunks=1, turns=1,
                later_text=0, steps=16, entry="layers")
    case.update(fields)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest model there is here, contiguous cache, everything in the L2: what a call costs
        _case("tiny_step", layers=2, q_heads=8, kv_heads=8, head_dim=64, paged=False, text_before=64, text_after=32,
              entry="step"),
        # one user waiting for tokens: 7B multi-head stack, short image prompt, the model's own layer loop
        _case("single_user_layers", steps=32),
        # the same stack serving a batch of 16
        _case("batch16_layers", batch=16, steps=32),
        # high-resolution images in tiles, batch of 8, the schedule of the repository's headline number
        _case("anyres_in_order", batch=8, visual=2880, text_after=93, entry="in_order"),
        # grouped-query stack, large batch, the model's own layer loop
        _case("gqa_batch32_layers", layers=28, q_heads=28, kv_heads=4, batch=32, visual=1024, text_after=61, steps=32),
        # long pruned video, few sequences, whole steps handed over at once
        _case("long_video_step", batch=4, visual=4096, text_after=221, entry="step"),
        # most layers lazy in blocks of four, no K kept in lazy layers
        _case("gla_blocks_layers", batch=8, visual=1920, text_after=93, lazy="blocks_of_4", mode="gla"),
        # sequences of different lengths, Eq. 8 as printed, inputs and outputs in host memory
        _case("ragged_host", batch=6, visual=1531, text_after=83, ragged=True, mode="vla_eq8", entry="host"),
        # time to the first token of a short image prompt
        _case("prompt_675", attend=True, steps=1, entry="step"),
        # the same for a long pruned video
        _case("prompt_4352", visual=4096, text_after=221, attend=True, steps=1, entry="step"),
        # a grouped-query prompt of odd length given in three pieces (chunked prefill)
        _case("gqa_prompt_chunks", layers=28, q_heads=28, kv_heads=4, visual=1397, text_after=61, attend=True, chunks=3,
              steps=1, entry="step"),
        # two turns of a conversation on a small stack with 64-wide heads
        _case("two_turns_d64", layers=12, q_heads=16, kv_heads=16, head_dim=64, batch=2, visual=577, text_after=40,
              attend=True, turns=2, later_text=45, steps=8, mode="gla", lazy="blocks_of_4"),
    ]


# A drawn case costs no more than the largest listed ones.
_MOST_PROMPT_BYTES = 12e9
_MOST_BYTES = 150e9
_MOST_FLOPS = 4.9e12


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    while True:
        attend = rng.random() < 0.4
        heads, kv_heads = rng.choice([(32, 32), (32, 32), (28, 4), (32, 8), (16, 16)])
        case = _case(
            None,
            layers=_log_int(rng, 6, 32), q_heads=heads, kv_heads=kv_heads,
            head_dim=64 if rng.random() < 0.1 else 128,
            batch=1 if attend and rng.random() < 0.7 else _log_int(rng, 1, 4 if attend else 32),
            text_before=rng.randint(1, 64), visual=_log_int(rng, 100, 4096), text_after=_log_int(rng, 16, 256),
            ragged=rng.random() < 0.4, lazy=rng.choice(["every_second", "every_second", "blocks_of_4"]),
            mode=rng.choice(["vla_qc", "vla_qc", "gla", "vla_eq8"]), attend=attend,
            chunks=rng.choice([1, 1, 2, 3]) if attend else 1,
            steps=rng.randint(1, 4) if attend else rng.randint(12, 32),
            entry=rng.choice(["step", "layers"] if attend else ["layers", "layers", "in_order", "step", "host"]))
        if attend and rng.random() < 0.25:
            case.update(turns=2, later_text=rng.randint(17, 90))
        w, prompt_bytes = _count(case)
        if prompt_bytes <= _MOST_PROMPT_BYTES and w["bytes"] <= _MOST_BYTES and w["flops"] <= _MOST_FLOPS:
            return case


# ---- sizes ----------------------------------------------------------------------------------


def _layer_kind(case):
    n = case["layers"]
    if case["lazy"] == "blocks_of_4":   # layers 0 and 1 ordinary, then one leader and three lazy layers
        return [1 if l >= 2 and (l - 2) % 4 else 0 for l in range(n)]
    return [1 if l % 2 and (l >= 3 or n == 2) else 0 for l in range(n)]


def _lengths(case):
    """(text before, visual, text after) of every sequence."""
    out = []
    for s in range(case["batch"]):
        f = 1.0 - 0.6 * (((s + 1) * 37) % 101) / 101.0 if case["ragged"] else 1.0
        out.append((case["text_before"], max(1, int(case["visual"] * f)), max(1, int(case["text_after"] * f))))
    return out


def _pieces(case, seq, turn):
    """Token kinds of a sequence's prompt in one turn, one array for each call that brings it."""
    if turn:
        return [np.zeros(case["later_text"], np.uint8)]
    before, visual, after = _lengths(case)[seq]
    kind = np.concatenate([np.zeros(before, np.uint8), np.ones(visual, np.uint8), np.zeros(after, np.uint8)])
    return [p for p in np.array_split(kind, case["chunks"]) if len(p)]


def _count(case):
    """Bytes and operations that a pass cannot do without, and the K/V bytes that its prompts bring."""
    n, hq, hkv, d = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"]
    lazy = sum(_layer_kind(case))
    full = n - lazy
    row, qrow = 2 * hkv * d, 2 * hq * d
    gla = case["mode"] == "gla"
    text_rows = n + (full if gla else n)     # layers that keep a text token's V and K
    vis_rows = n + full
    score_layers = full if gla else n
    bytes_ = flops = prompt = 0.0
    for s in range(case["batch"]):
        text = vis = 0
        for turn in range(case["turns"]):
            for kind in _pieces(case, s, turn):
                nv = int(kind.sum())
                nt = len(kind) - nv
                new = nt * text_rows + nv * vis_rows
                prompt += 2.0 * n * len(kind) * row
                bytes_ += 2.0 * new * row                                      # read from the caller, stored
                if case["attend"]:
                    pairs = 0.5 * len(kind) * (len(kind) + 1) + len(kind) * (text + vis)
                    flops += 2.0 * d * hq * pairs * (score_layers + n)
                    bytes_ += (nt * (full if gla else n) + nv * full + len(kind) * n) * qrow   # queries, outputs
                    bytes_ += (text * text_rows + vis * vis_rows) * row        # what the cache holds already
                text, vis = text + nt, vis + nv
            for _ in range(case["steps"]):
                text += 1
                rows = text * text_rows + vis * vis_rows
                bytes_ += rows * row + text_rows * row + 2.0 * n * qrow
                flops += 2.0 * d * hq * (text + vis) * (score_layers + n)
    return {"bytes": bytes_, "flops": flops}, prompt


def work(case):
    return _count(case)[0]


def tolerance(case):
    # Four times what the library's own schedules and chunk sizes differ by on the same inputs (fp32
    # sums in another order, then one bf16 rounding of the output: rel 4.6e-5, max 7.8e-3), and four
    # times what its two prompt kernels differ by where softmax weights are rounded to bf16 as well
    # (prompts, grouped queries: rel 2.1e-3, in a prompt's later chunks 3e-3; max 2.9e-2).
    if case["attend"] or case["q_heads"] != case["kv_heads"]:
        return {"rel": 1e-2, "max": 1.2e-1}
    return {"rel": 2e-4, "max": 3.2e-2}


# ---- a pass ---------------------------------------------------------------------------------


def _inputs(case, seed):
    """Per turn the calls that bring its prompts (sequences, kinds, tensors by name), and q, k, v of the decode steps."""
    n, hq, hkv, d, b = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"], case["batch"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)

    prompts = []
    for turn in range(case["turns"]):
        if not case["attend"]:
            kinds = [_pieces(case, s, turn)[0] for s in range(b)]
            total = sum(len(kind) for kind in kinds)
            prompts.append([(list(range(b)), kinds, {"k": normal(n, total, hkv, d), "v": normal(n, total, hkv, d)})])
            continue
        calls = []
        for s in range(b):
            for kind in _pieces(case, s, turn):
                t = len(kind)
                calls.append(([s], [kind], {"q": normal(n, t, hq, d), "k": normal(n, t, hkv, d),
                                            "v": normal(n, t, hkv, d)}))
        prompts.append(calls)
    q, k, v = (normal(case["turns"], case["steps"], n, b, h, d) for h in (hq, hkv, hkv))
    return prompts, q, k, v


def prepare(case, seed):
    n, hq, hkv, d, b = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"], case["batch"]
    turns, steps = case["turns"], case["steps"]
    lens = _lengths(case)
    text = [before + after + (turns - 1) * case["later_text"] + turns * steps for before, _, after in lens]
    vis = [v for _, v, _ in lens]
    pages = sum(2 * n * ((t + 15) // 16 + (v + 15) // 16) for t, v in zip(text, vis)) + 16
    session = Session(n, hq, hkv, d, _layer_kind(case), page_size=16 if case["paged"] else 0, max_seqs=b,
                      max_tokens_per_seq=max(text + vis), n_pages=pages if case["paged"] else 0,
                      lazy_mode=MODES[case["mode"]])
    if case["entry"] == "in_order":
        session.set_option("in_order_launches", 1)

    drawn, q, k, v = _inputs(case, seed)
    prompts = []   # per turn: the arguments of the calls that bring its prompts
    for calls in drawn:
        if case["attend"]:
            prompts.append([(ids[0], kinds[0], t["q"], t["k"], t["v"], torch.empty_like(t["q"]))
                            for ids, kinds, t in calls])
        else:
            prompts.append([(ids, [len(kind) for kind in kinds], np.concatenate(kinds), t["k"], t["v"])
                            for ids, kinds, t in calls])

    out = torch.empty(turns, steps, n, b, hq, d, device="cuda", dtype=torch.bfloat16)
    if case["entry"] == "host":
        q, k, v, out = (t.cpu().pin_memory() for t in (q, k, v, out))
    per_step = [[tuple(x[turn, i] for x in (q, k, v, out)) for i in range(steps)] for turn in range(turns)]
    if case["entry"] == "layers":   # a layer's own tensors, as a model's loop has them
        per_step = [[[tuple(x[l] for x in tensors) for l in range(n)] for tensors in turn] for turn in per_step]
    return {"case": case, "session": session, "ids": list(range(b)), "prompts": prompts, "steps": per_step, "out": out}


def run(state):
    case, session, ids = state["case"], state["session"], state["ids"]
    entry = case["entry"]
    for prompts, steps in zip(state["prompts"], state["steps"]):
        for call in prompts:
            if case["attend"]:
                session.prefill_attend(*call)
            else:
                session.prefill_append(*call)
        for tensors in steps:
            if entry == "layers":
                session.decode_begin(ids)
                for layer, (q, k, v, out) in enumerate(tensors):
                    session.decode_layer(layer, q, k, v, out)
            elif entry == "host":
                session.decode_step_host(ids, *tensors)
            else:
                session.decode_step(ids, *tensors)
    for s in reversed(ids):
        qc.qc_free_seq(session.cache, s)
    outputs = [state["out"]]
    if case["attend"]:
        outputs += [call[-1] for prompts in state["prompts"] for call in prompts]
    return outputs


# ---- the same in 64 bits --------------------------------------------------------------------


def _attention(q, q_visual, k, v, visual):
    """Softmax attention of the last len(q) tokens of k and v, each over the tokens up to itself.

    q: [new][hq][d]; k, v: [tokens][hkv][d]; where ``q_visual`` is given it scores the visual keys."""
    new, hq, d = q.shape
    tokens, hkv, _ = k.shape
    group = hq // hkv
    out = torch.empty_like(q)
    at = torch.arange(tokens, device=q.device)
    hidden = (at[None, :] > at[tokens - new:, None]).repeat(group, 1)          # [group * new][tokens]
    step = max(1, int(2 ** 27 // (group * new * tokens)))
    for h in range(0, hkv, step):
        e = min(hkv, h + step)

        def scores(x):
            x = x[:, h * group:e * group].reshape(new, e - h, group, d).permute(1, 2, 0, 3).reshape(e - h, group * new, d)
            return x @ k[:, h:e].permute(1, 2, 0)

        s = scores(q)
        if q_visual is not None:
            s = torch.where(visual, scores(q_visual), s)
        w = (s * d ** -0.5).masked_fill_(hidden, float("-inf")).softmax(-1)
        o = (w @ v[:, h:e].permute(1, 0, 2)).reshape(e - h, group, new, d)
        out[:, h * group:e * group] = o.permute(2, 0, 1, 3).reshape(new, (e - h) * group, d)
    return out


def exact(case, seed):
    """Lazy attention written down directly: a lazy layer's queries and keys are its leader's, of all
    tokens (gla) or of the visual ones; a generated token is text, and its query on visual keys is
    the leader's in vla_qc, its own in vla_eq8."""
    drawn, q, k, v = _inputs(case, seed)
    n, steps, gla = case["layers"], case["steps"], case["mode"] == "gla"
    kinds = _layer_kind(case)
    leader = [max(x for x in range(l + 1) if not kinds[x]) for l in range(n)]
    out = torch.empty(case["turns"], steps, n, case["batch"], case["q_heads"], case["head_dim"], device="cuda",
                      dtype=torch.float64)
    prompt_outs = [[torch.empty(t["q"].shape, device="cuda", dtype=torch.float64) for _, _, t in calls]
                   if case["attend"] else [] for calls in drawn]
    for s in range(case["batch"]):
        for l in range(n):
            c = leader[l]
            keys, values, vis = [], [], []

            def add(kind, key, key_lead, value):
                visual = torch.from_numpy(kind != 0).cuda()
                keys.append((key_lead if gla else torch.where(visual[:, None, None], key_lead, key)).double())
                values.append(value.double())
                vis.append(visual)
                return torch.cat(keys), torch.cat(values), torch.cat(vis)

            for turn, calls in enumerate(drawn):
                for i, (ids, call_kinds, t) in enumerate(calls):
                    if s not in ids:
                        continue
                    first = sum(len(x) for x in call_kinds[:ids.index(s)])
                    kind = call_kinds[ids.index(s)]
                    part = {name: x[:, first:first + len(kind)] for name, x in t.items()}
                    kv = add(kind, part["k"][l], part["k"][c], part["v"][l])
                    if case["attend"]:
                        own = part["q"][c] if gla else torch.where(kv[2][-len(kind):, None, None], part["q"][c], part["q"][l])
                        prompt_outs[turn][i][l] = _attention(own.double(), None, *kv)
                kv = add(np.zeros(steps, np.uint8), k[turn, :, l, s], k[turn, :, c, s], v[turn, :, l, s])
                lead_q = q[turn, :, c, s].double()
                own_q = lead_q if gla else q[turn, :, l, s].double()
                out[turn, :, l, s] = _attention(own_q, lead_q if case["mode"] == "vla_qc" else None, *kv)
    return [out] + [x for outs in prompt_outs for x in outs]
