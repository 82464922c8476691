"""What is measured of the framework's speed: calls of its public entry points as a serving program makes them.

A case is a dict of plain values.  ``kind`` names the entry point:

* ``score``     apack_score: relevance scores of one pruning layer's keys
* ``select``    apack_select: top-k of given scores and the ordered keep map
* ``compact``   apack_compact: slices the K/V caches and the hidden states, out of place or in place
* ``step``      apack_prune_step: score, select and compact in one call
* ``schedule``  ProgressivePrune.run: a progressive schedule in one call
* ``decode``    apack_decode_attention: one decode token per sequence over the (compacted) caches
* ``align``     apack_frame_alignment: windowed CKA and gate of the pre-LLM stage

Sequences are laid out as in the workloads: system tokens, then per second the video frames (2 per
second, ``tpf`` tokens each) and 25 audio tokens, then the query span.  A batch draws every
sequence's length and query rows from the case's ranges with its ``layout`` number, so the shapes
belong to the case and the values to the seed.
"""

import math
import random

import numpy as np
import torch

import paper_2608_08794_gb300 as ap
from paper_2608_08794_gb300.schedule import ProgressivePrune

D = 128
N_SYS = 16
AUDIO_PER_SECOND = 25
FPS = 2
HEADS = ("28/4", "16/2", "32/8", "8/8", "12/2")
SCORE_KINDS = ("score", "step", "schedule")


def listed():
    return [
        # The smallest step: a 10-second clip, one layer's cache, a 32-token question.  Seven small
        # kernels in a row: launches and latency.
        dict(name="step_10s", kind="step", heads="28/4", hidden=3584, seqs=1, seconds_lo=10, seconds_hi=10, tpf=50,
             q_lo=32, q_hi=32, domain="mm", mode="modality", keep=0.36, layers=1, layout=1),
        # The last step of the paper's schedule (the last query token scores, one top-k over all
        # multimodal tokens, the last layer only): as small as a step of a long video gets.
        dict(name="step_last_layer", kind="step", heads="28/4", hidden=3584, seqs=1, seconds_lo=72, seconds_hi=72,
             tpf=101, q_lo=1, q_hi=1, domain="mm", mode="joint", keep=0.85, layers=1, layout=2),
        # A one-minute clip in a 3B-shaped model, scored over the decoder's own causal rows.
        dict(name="score_1min_causal", kind="score", heads="16/2", seqs=1, seconds_lo=60, seconds_hi=60, tpf=60,
             q_lo=64, q_hi=64, domain="causal", layout=3),
        # The benchmark's sequence: ten minutes of video, a 256-token query span.
        dict(name="score_10min", kind="score", heads="28/4", seqs=1, seconds_lo=600, seconds_hi=600, tpf=100,
             q_lo=256, q_hi=256, domain="mm", layout=4),
        # A serving batch of 16 clips of half a minute to five minutes with questions of any length.
        dict(name="score_ragged16", kind="score", heads="28/4", seqs=16, seconds_lo=30, seconds_hi=300, tpf=100,
             q_lo=16, q_hi=256, domain="mm", layout=5),
        # The paper's own scoring (the last query token) of the ten-minute sequence.
        dict(name="score_10min_last_query", kind="score", heads="28/4", seqs=1, seconds_lo=600, seconds_hi=600,
             tpf=100, q_lo=1, q_hi=1, domain="mm", layout=6),
        # A short command of three tokens about a five-minute clip.
        dict(name="score_short_query", kind="score", heads="28/4", seqs=1, seconds_lo=300, seconds_hi=300, tpf=100,
             q_lo=3, q_hi=3, domain="mm", layout=7),
        # The keep map of the ten-minute sequence, jointly over both modalities.
        dict(name="select_10min", kind="select", seqs=1, seconds_lo=600, seconds_hi=600, tpf=100, mode="joint",
             keep=0.45, layout=8),
        # A cache that has no room for a second copy: 24 layers and the hidden states of the
        # ten-minute sequence sliced within their own buffers.
        dict(name="compact_in_place_10min", kind="compact", heads="28/4", hidden=3584, layers=24, seqs=1,
             seconds_lo=600, seconds_hi=600, tpf=100, keep=0.43, in_place=True, layout=9),
        # The three-step schedule of the two-minute clip, through the class a serving program keeps.
        dict(name="schedule_2min", kind="schedule", heads="28/4", hidden=3584, layers=28, prune="4,12,20",
             keep="0.43,0.28,0.17", seqs=1, seconds_lo=120, seconds_hi=120, tpf=100, q_lo=128, q_hi=128, domain="mm",
             mode="modality", layout=10),
        # One decode step of a batch over pruned caches of clips of many lengths.
        dict(name="decode_batch16", kind="decode", heads="28/4", seqs=16, len_lo=600, len_hi=12000, layout=11),
        # The pre-LLM alignment of the ten-minute clip (1200 frames of 100 tokens).
        dict(name="align_10min", kind="align", frames=1200, tpf=100, dim=3584, window=3, layout=12),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges; costs stay below the largest listed ones."""
    kind = rng.choice(("score", "score", "score", "select", "compact", "step", "step", "schedule", "decode", "decode",
                       "align"))
    layout = rng.randrange(1 << 20)
    heads = rng.choice(("28/4", "28/4", "16/2") + HEADS)
    hidden = {"28/4": 3584, "16/2": 2048}.get(heads, 4096)
    if kind == "align":
        return dict(kind=kind, frames=_log_uniform(rng, 8, 1200), tpf=_log_uniform(rng, 25, 100),
                    dim=rng.choice((3584, 2048, 1280, 1000)), window=rng.choice((3, 3, 5, 7)), layout=layout)
    seqs = rng.choice((1, 1, 1, rng.randint(2, 16)))
    if kind == "decode":
        hi = _log_uniform(rng, 200, 135000 // seqs)
        return dict(kind=kind, heads=rng.choice((heads, "8/1")), seqs=seqs, len_lo=max(1, hi // 8), len_hi=hi,
                    layout=layout)
    hi = _log_uniform(rng, 4, 600 if seqs == 1 else 120)
    lo = hi if seqs == 1 else max(2, hi // 4)
    tpf = rng.choice((100, 60, rng.randint(25, 100)))
    base = dict(kind=kind, seqs=seqs, seconds_lo=lo, seconds_hi=hi, tpf=tpf, layout=layout)
    keep = round(rng.uniform(0.1, 0.9), 3)
    mode = rng.choice(("modality", "joint"))
    if kind == "select":
        return dict(base, mode=mode, keep=keep)
    if seqs == 1:
        q_hi = rng.choice((1, 1, _log_uniform(rng, 2, 256), _log_uniform(rng, 2, 256)))
        q_lo = q_hi
    else:
        # a batch: the models' own heads, the last query token or questions of 16 tokens and more
        heads = rng.choice(("28/4", "16/2"))
        hidden = {"28/4": 3584, "16/2": 2048}[heads]
        q_hi = rng.choice((1, _log_uniform(rng, 64, 256)))
        q_lo = max(1, q_hi // 4)
    rows = dict(q_lo=q_lo, q_hi=q_hi, domain=rng.choice(("mm", "mm", "causal")))
    if kind == "score":
        return dict(base, heads=heads, **rows)
    # caches: at most the compaction listed above (24 layers of 135,000 tokens of 1 KB rows)
    tokens = hi * (FPS * tpf + AUDIO_PER_SECOND) * seqs
    row = 2 * D * int(heads.split("/")[1])
    most = max(1, min(28, int(2.5e9 // (tokens * row))))
    if kind == "compact":
        return dict(base, heads=heads, hidden=hidden, layers=rng.randint(1, most), keep=keep,
                    in_place=rng.random() < 0.5)
    if kind == "step":
        return dict(base, heads=heads, hidden=hidden, layers=rng.randint(1, most), mode=mode, keep=keep, **rows)
    steps = rng.randint(2, 3)
    layers = max(steps, most)
    prune = sorted(rng.sample(range(layers), steps))
    kept = sorted((round(rng.uniform(0.12, 0.8), 3) for _ in range(steps)), reverse=True)
    return dict(base, heads=heads, hidden=hidden, layers=layers, prune=",".join(map(str, prune)),
                keep=",".join(map(str, kept)), mode=mode, **rows)


# ---------------------------------------------------------------- shapes


class Shape:
    """Host-side layout of a case's batch: offsets, query rows, modality codes, counts."""

    def __init__(self, case):
        r = random.Random(case["layout"])
        B = case["seqs"]
        seconds = [r.randint(case["seconds_lo"], case["seconds_hi"]) for _ in range(B)]
        nq = [r.randint(case.get("q_lo", 1), case.get("q_hi", 1)) for _ in range(B)]
        tpf = case["tpf"]
        second = np.concatenate([np.full(FPS * tpf, ap.APACK_MOD_VISUAL, np.uint8),
                                 np.full(AUDIO_PER_SECOND, ap.APACK_MOD_AUDIO, np.uint8)])
        mods = [np.concatenate([np.zeros(N_SYS, np.uint8), np.tile(second, s), np.zeros(n, np.uint8)])
                for s, n in zip(seconds, nq)]
        self.B, self.nq = B, nq
        self.len = [m.size for m in mods]
        self.modality = np.concatenate(mods)
        self.cu = np.concatenate([[0], np.cumsum(self.len)]).astype(np.int32)
        self.cuq = np.concatenate([[0], np.cumsum(nq)]).astype(np.int32)
        self.n_audio = np.array([AUDIO_PER_SECOND * s for s in seconds], np.int32)
        self.n_visual = np.array([FPS * tpf * s for s in seconds], np.int32)
        self.T = int(self.cu[-1])


def _heads(case):
    hq, hkv = case["heads"].split("/")
    return int(hq), int(hkv)


def _mode(case):
    return ap.APACK_SELECT_JOINT if case["mode"] == "joint" else ap.APACK_SELECT_PER_MODALITY


def _domain(case):
    return ap.APACK_SOFTMAX_CAUSAL_ROW if case.get("domain") == "causal" else ap.APACK_SOFTMAX_MM


def _ratios(case):
    return [float(x) for x in str(case["keep"]).split(",")]


def _counts(case, shape):
    """Keep counts [B, 2] after every step (cumulative ratios over the counts entering step 0)."""
    s = ap.Seqs(shape.cu, shape.cuq, shape.n_audio, shape.n_visual, torch.empty(1, dtype=torch.uint8), 1, 1)
    out = []
    for r in _ratios(case):
        ratio = np.full((shape.B, 2), r, np.float32)
        if case["mode"] == "modality":
            ratio[:, 0] = min(1.0, 1.2 * r)          # audio keeps a little more than video
        out.append(ap.apack_keep_counts(s, ratio, _mode(case))[0])
    return out


def _lengths(case):
    r = random.Random(case["layout"])
    return [_log_uniform(r, case["len_lo"], case["len_hi"]) for _ in range(case["seqs"])]


# ---------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, *shape, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=g)


def _ws(nbytes):
    raw = torch.zeros(nbytes + 256, dtype=torch.uint8, device="cuda")
    off = (-raw.data_ptr()) % 256
    return raw[off:off + nbytes]


def _strength(case, shape, g, counts):
    """How strongly each token answers the query, in [0, 1].  Scoring alone: 5 % of the tokens
    moderately, 0.1 % strongly (a heavy tail).  With a selection: the tokens that each step keeps
    stand one level above those it drops, so that the order of two nearly equal scores decides
    nothing."""
    T = shape.T
    out = torch.zeros(T, device="cuda")
    noise = torch.rand(T, generator=g, device="cuda")
    if counts is None:
        out[noise < 0.05] = 0.5
        out[noise < 0.001] = 1.0
        return out
    mod = torch.from_numpy(shape.modality).cuda()
    for b in range(shape.B):
        t0, t1 = int(shape.cu[b]), int(shape.cu[b + 1])
        joint = case["mode"] == "joint"
        for m in range(1 if joint else 2):
            seg = mod[t0:t1] > 0 if joint else mod[t0:t1] == m + 1
            idx = seg.nonzero().view(-1) + t0
            order = idx[torch.argsort(noise[idx])]
            for k in counts:
                out[order[:int(k[b, m])]] += 1.0 / len(counts)
    return out


def _queries_and_keys(case, shape, g, levels, strength, keys):
    """Query rows [sum n_q, Hq, D], and `keys` (one layer's K, [T, Hkv, D]) rewritten in place: both
    normal, with a per-(sequence, KV head) direction that the queries share and the tokens that
    answer them lean towards (4 in the logit per level)."""
    hq, hkv = _heads(case)
    u = torch.nn.functional.normalize(_normal(g, shape.B, hkv, D, dtype=torch.float32), dim=-1)
    q = _normal(g, int(shape.cuq[-1]), hq, D, dtype=torch.float32)
    for b in range(shape.B):
        rows = slice(int(shape.cuq[b]), int(shape.cuq[b + 1]))
        ub = u[b].repeat_interleave(hq // hkv, 0)
        q[rows] += (4.0 * levels - (q[rows] * ub).sum(-1, keepdim=True)) * ub
        t = slice(int(shape.cu[b]), int(shape.cu[b + 1]))
        k = keys[t].float()
        k += (math.sqrt(D) * strength[t].view(-1, 1, 1) - (k * u[b]).sum(-1, keepdim=True)) * u[b]
        keys[t] = k.to(torch.bfloat16)
    return q.to(torch.bfloat16)


def _seqs(case, shape, modality):
    hq, hkv = _heads(case)
    return ap.Seqs(shape.cu, shape.cuq, shape.n_audio, shape.n_visual, modality, hq, hkv,
                   softmax_domain=_domain(case))


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, _gen(seed))


def _prepare_score(case, g):
    shape = Shape(case)
    hkv = _heads(case)[1]
    k = _normal(g, shape.T, hkv, D)
    q = _queries_and_keys(case, shape, g, 1, _strength(case, shape, g, None), k)
    mod = torch.from_numpy(shape.modality).cuda()
    seqs = _seqs(case, shape, mod)
    return dict(case=case, shape=shape, seqs=seqs, q=q, k=k, mod=mod, scores=torch.empty(shape.T, device="cuda"),
                ws=_ws(ap.apack_workspace_size(seqs)))


def _prepare_select(case, g):
    shape = Shape(case)
    mod = torch.from_numpy(shape.modality).cuda()
    # relevance scores span decades and sum to about 1 per sequence; some tokens tie
    s = torch.exp(1.3 * _normal(g, shape.T, dtype=torch.float32)) / (shape.T / shape.B)
    s[torch.rand(shape.T, generator=g, device="cuda") < 0.01] = 0.5 * shape.B / shape.T
    s[mod == 0] = 0.0
    hq, hkv = 28, 4
    seqs = ap.Seqs(shape.cu, shape.cuq, shape.n_audio, shape.n_visual, mod, hq, hkv)
    counts = _counts(case, shape)[0]
    n_out = int(shape.T - (shape.n_audio + shape.n_visual).sum() + counts.sum())
    return dict(case=case, shape=shape, seqs=seqs, scores=s, mod=mod, counts=counts, mode=_mode(case),
                keep=torch.empty(n_out, dtype=torch.int32, device="cuda"),
                mod_out=torch.empty(n_out, dtype=torch.uint8, device="cuda"),
                new_cu=torch.empty(shape.B + 1, dtype=torch.int32, device="cuda"),
                ws=_ws(ap.apack_workspace_size(seqs)))


def _kept(case, shape, g):
    """Ascending kept rows: every text token, and about the keep ratio of the others."""
    keep = torch.rand(shape.T, generator=g, device="cuda") < float(case["keep"])
    keep |= torch.from_numpy(shape.modality).cuda() == 0
    return keep.nonzero().view(-1).to(torch.int32)


def _prepare_compact(case, g):
    shape = Shape(case)
    hkv = _heads(case)[1]
    L, T, row = case["layers"], shape.T, hkv * D * 2
    # the number of kept rows is the case's, which rows the seed's
    idx = _kept(case, shape, _gen(case["layout"]))
    n = idx.numel()
    pick = torch.rand(T, generator=g, device="cuda").argsort()[:n]
    idx = pick.sort().values.to(torch.int32)
    src = [_normal(g, L, T, hkv, D), _normal(g, L, T, hkv, D), _normal(g, T, case["hidden"])]
    if case["in_place"]:
        dst = src
        stride = T * row
    else:
        dst = [torch.empty(L, n, hkv, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        dst.append(torch.empty(n, case["hidden"], dtype=torch.bfloat16, device="cuda"))
        stride = n * row
    planes = [ap.make_plane(src[0], dst[0], row, L, T * row, stride), ap.make_plane(src[1], dst[1], row, L, T * row, stride),
              ap.make_plane(src[2], dst[2], case["hidden"] * 2)]
    return dict(case=case, shape=shape, idx=idx, n=n, src=src, dst=dst, planes=planes, ws=_ws(1024))


def _prepare_step(case, g):
    shape = Shape(case)
    hkv = _heads(case)[1]
    L, T = case["layers"], shape.T
    counts = _counts(case, shape)
    k, v, h = _normal(g, L, T, hkv, D), _normal(g, L, T, hkv, D), _normal(g, T, case["hidden"])
    q = _queries_and_keys(case, shape, g, 1, _strength(case, shape, g, counts), k[0])
    mod = torch.from_numpy(shape.modality).cuda()
    seqs = _seqs(case, shape, mod)
    n = int(T - (shape.n_audio + shape.n_visual).sum() + counts[0].sum())

    def out(*s, dtype=torch.bfloat16):
        return torch.empty(s, dtype=dtype, device="cuda")

    return dict(case=case, shape=shape, seqs=seqs, q=q, k=k, v=v, h=h, mod=mod, counts=counts[0], n=n, mode=_mode(case),
                k_out=out(L, n, hkv, D), v_out=out(L, n, hkv, D), h_out=out(n, case["hidden"]),
                mod_out=out(n, dtype=torch.uint8), keep=out(n, dtype=torch.int32), scores=out(T, dtype=torch.float32),
                ws=_ws(ap.apack_workspace_size(seqs)))


def _prepare_schedule(case, g):
    shape = Shape(case)
    hq, hkv = _heads(case)
    layers = [int(x) for x in case["prune"].split(",")]
    counts = _counts(case, shape)
    pp = ProgressivePrune(shape.cu, shape.cuq, shape.n_audio, shape.n_visual, hq, hkv, case["layers"], case["hidden"],
                          layers, counts, select_mode=_mode(case), softmax_domain=_domain(case))
    pp.k_in.normal_(generator=g)
    pp.v_in.normal_(generator=g)
    pp.hidden_in.normal_(generator=g)
    pp.modality_in.copy_(torch.from_numpy(shape.modality))
    strength = _strength(case, shape, g, counts)
    for i, l in enumerate(layers):
        pp.q[i].copy_(_queries_and_keys(case, shape, g, len(layers), strength, pp.k_in[l - layers[0]]))
    return dict(case=case, shape=shape, pp=pp, counts=counts, layers=layers)


def _prepare_decode(case, g):
    hq, hkv = _heads(case)
    lens = _lengths(case)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    T = int(cu[-1])
    q = 1.5 * _normal(g, len(lens), hq, D, dtype=torch.float32)     # a mildly peaked attention row
    return dict(case=case, cu=cu, q=q.to(torch.bfloat16), k=_normal(g, T, hkv, D), v=_normal(g, T, hkv, D),
                out=torch.empty(len(lens), hq, D, device="cuda"), ws=_ws(ap.apack_decode_workspace_size(cu, hq, hkv)))


def _prepare_align(case, g):
    F, tpf, dim = case["frames"], case["tpf"], case["dim"]
    n_audio = max(F, F * AUDIO_PER_SECOND // FPS)
    # embeddings drift in a few directions, slowly within a scene and fast at cuts; the audio
    # follows the picture in part
    pace = torch.exp(1.5 * _normal(g, F, 1, dtype=torch.float32))
    step_v = pace * _normal(g, F, 8, dtype=torch.float32)
    pace_a = torch.exp(1.5 * _normal(g, F, 1, dtype=torch.float32))
    step_a = pace_a * _normal(g, F, 8, dtype=torch.float32)
    basis = 0.05 * _normal(g, 16, dim, dtype=torch.float32)
    lat_v = step_v.cumsum(0) @ basis[:8]
    lat_a = step_a.cumsum(0) @ basis[8:]
    visual = (_normal(g, F, tpf, dim, dtype=torch.float32) + lat_v[:, None]).to(torch.bfloat16).view(F * tpf, dim)
    at = (torch.arange(n_audio, device="cuda") * F) // n_audio
    audio = (_normal(g, n_audio, dim, dtype=torch.float32) + lat_a[at]).to(torch.bfloat16)

    def out(n):
        return torch.empty(n, device="cuda")

    return dict(case=case, visual=visual, audio=audio, n_audio=n_audio, c=out(F), s=out(F), dn=out(F), cbar=out(1),
                ws=_ws(ap.apack_frame_alignment_workspace_size(F, dim)))


# ---------------------------------------------------------------- one pass


def run(s):
    return globals()["_run_" + s["case"]["kind"]](s)


def _run_score(s):
    ap.apack_score(s["seqs"], s["q"], s["k"], s["seqs"].struct.num_kv_heads * D * 2, s["scores"], s["ws"])
    return s["scores"]


def _run_select(s):
    ap.apack_select(s["seqs"], s["scores"], s["counts"], s["keep"], s["ws"], select_mode=s["mode"],
                    modality_out=s["mod_out"], new_cu_seqlens=s["new_cu"])
    return dict(keep=s["keep"], modality=s["mod_out"], cu=s["new_cu"])


def _run_compact(s):
    ap.apack_compact(s["idx"], s["n"], s["planes"], ws=s["ws"])
    return [t[..., :s["n"], :] if t.dim() == 2 else t[:, :s["n"]] for t in s["dst"]]


def _run_step(s):
    c = s["case"]
    row = s["k"].shape[2] * D * 2
    cu = ap.apack_prune_step(s["seqs"], 28 - c["layers"], 28, s["q"], s["k"], s["v"], s["shape"].T * row, s["h"],
                             c["hidden"], keep_count=s["counts"], select_mode=s["mode"], k_out=s["k_out"],
                             v_out=s["v_out"], kv_out_layer_stride=s["n"] * row, hidden_out=s["h_out"],
                             modality_out=s["mod_out"], keep_idx=s["keep"], scores=s["scores"], ws=s["ws"])
    return dict(scores=s["scores"], keep=s["keep"], modality=s["mod_out"], k=s["k_out"], v=s["v_out"],
                hidden=s["h_out"], cu=cu)


def _run_schedule(s):
    pp = s["pp"]
    pp.run()
    last = len(s["layers"]) - 1
    k, v = pp.output_kv(last)
    k1, v1 = pp.output_kv(last - 1)                  # the other of the two buffers that alternate
    return dict(scores=pp.scores[:pp.t_out[last - 1]], keep=pp.keep_idx, modality=pp.mod_out[last % 2][:pp.t_out[last]],
                k=k, v=v, k_before=k1, v_before=v1, hidden=pp.output_hidden(last), cu=pp.new_cu)


def _run_decode(s):
    hq, hkv = _heads(s["case"])
    ap.apack_decode_attention(s["cu"], s["q"], s["k"], s["v"], hkv * D * 2, hq, hkv, s["out"], s["ws"])
    return s["out"]


def _run_align(s):
    c = s["case"]
    ap.apack_frame_alignment(s["visual"], s["audio"], c["frames"], c["tpf"], s["n_audio"], c["dim"], s["c"], s["s"],
                             s["ws"], window=c["window"], dnorm_out=s["dn"], cbar_out=s["cbar"])
    return dict(c=s["c"], s=s["s"], dnorm=s["dn"], cbar=s["cbar"])


# ---------------------------------------------------------------- what a pass cannot do without


def _score_work(lens, nq, hq, hkv):
    flops = sum(2.0 * D * hq * n * q for n, q in zip(lens, nq))
    nbytes = sum(n * (hkv * D * 2 + 1 + 4) + q * hq * D * 2 for n, q in zip(lens, nq))
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "align":
        F = case["frames"]
        n = F * case["tpf"] + max(F, F * AUDIO_PER_SECOND // FPS)
        return {"bytes": n * case["dim"] * 2 + 12 * F, "flops": n * case["dim"]}
    hq, hkv = _heads(case) if "heads" in case else (28, 4)
    row = hkv * D * 2
    if kind == "decode":
        T = sum(_lengths(case))
        return {"bytes": 2 * T * row + case["seqs"] * hq * D * 6, "flops": 4.0 * D * hq * T}
    shape = Shape(case)
    if kind == "score":
        b, f = _score_work(shape.len, shape.nq, hq, hkv)
        return {"bytes": b, "flops": f}
    if kind == "compact":
        n = _kept(case, shape, _gen(case["layout"])).numel()
        return {"bytes": 2 * n * (2 * case["layers"] * row + 2 * case["hidden"]) + 4 * n, "flops": 0}
    other = shape.T - int((shape.n_audio + shape.n_visual).sum())
    n_after = [other + int(k.sum()) for k in _counts(case, shape)]
    if kind == "select":
        return {"bytes": 5 * shape.T + 5 * n_after[0] + 4 * (shape.B + 1), "flops": 0}
    b = f = 0.0
    counts = _counts(case, shape)
    text = np.array(shape.len) - shape.n_audio - shape.n_visual
    entering = [np.array(shape.len)] + [text + k.sum(1) for k in counts]
    layers = [int(x) for x in case["prune"].split(",")] if kind == "schedule" else [0]
    for i, l in enumerate(layers):
        sb, sf = _score_work(entering[i].tolist(), shape.nq, hq, hkv)
        n, planes = n_after[i], 2 * (case["layers"] - l)
        b += sb + int(entering[i].sum()) + 5 * n + 2 * n * (planes * row + 2 * case["hidden"])
        f += sf
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Four times the largest difference from `exact` seen over the listed and some drawn cases."""
    kind = case["kind"]
    if kind in ("select", "compact"):
        return "exact"
    if kind in SCORE_KINDS:
        # fp32 sums of fp32 exponentials, 1e5 of them per row; copied rows are equal
        return {"rel": 1.5e-6, "max": 2e-5, "differ": 0.0}
    if kind == "decode":
        # probabilities carried as bf16 pairs
        return {"rel": 1e-5, "max": 1e-4}
    # sums of bf16 rows in fp32, then differences of neighbouring frames' means
    return {"rel": 1e-6, "max": 1e-4}


# ---------------------------------------------------------------- the same in 64 bits


def _exact_scores(q, k, modality, cu, cuq, causal):
    """Relevance scores in 64 bits: q [n, Hq, D], k [T, Hkv, D], modality [T] on the GPU."""
    hq, hkv = q.shape[1], k.shape[1]
    G = hq // hkv
    out = torch.zeros(k.shape[0], dtype=torch.float64, device="cuda")
    for b in range(len(cu) - 1):
        t = slice(int(cu[b]), int(cu[b + 1]))
        nq, n = int(cuq[b + 1] - cuq[b]), int(cu[b + 1] - cu[b])
        if nq == 0 or n == 0:
            continue
        mm = modality[t] > 0
        pos = torch.arange(n, device="cuda")
        for g in range(hkv):
            kg = k[t, g].double()
            for j in range(G):
                qg = q[int(cuq[b]):int(cuq[b + 1]), g * G + j].double()
                x = qg @ kg.T / math.sqrt(D)
                if causal:
                    x.masked_fill_(pos[None, :] > (n - nq + torch.arange(nq, device="cuda"))[:, None], -math.inf)
                else:
                    x.masked_fill_(~mm[None, :], -math.inf)
                out[t] += torch.softmax(x, -1).sum(0) * mm
        out[t] /= hq * nq
    return out


def _exact_keep(scores, modality, cu, counts, joint):
    """Kept rows in order, and the offsets after the step."""
    keep = modality == 0
    for b in range(len(cu) - 1):
        t0, t1 = int(cu[b]), int(cu[b + 1])
        for m in range(1 if joint else 2):
            seg = modality[t0:t1] > 0 if joint else modality[t0:t1] == m + 1
            idx = seg.nonzero().view(-1) + t0
            order = idx[torch.sort(scores[idx], descending=True, stable=True).indices]
            keep[order[:int(counts[b, m])]] = True
    kept = keep.nonzero().view(-1)
    new = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), keep.cumsum(0)])[torch.as_tensor(cu, device="cuda").long()]
    return kept, new


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "score":
        sh = s["shape"]
        return _exact_scores(s["q"], s["k"], s["mod"], sh.cu, sh.cuq, case["domain"] == "causal")
    if kind == "select":
        kept, new = _exact_keep(s["scores"], s["mod"], s["shape"].cu, s["counts"], case["mode"] == "joint")
        return dict(keep=kept.int(), modality=s["mod"][kept], cu=new.int())
    if kind == "compact":
        idx = s["idx"].long()
        return [t[..., idx, :] if t.dim() == 2 else t[:, idx] for t in s["src"]]
    if kind == "step":
        sh = s["shape"]
        sc = _exact_scores(s["q"], s["k"][0], s["mod"], sh.cu, sh.cuq, case["domain"] == "causal")
        kept, new = _exact_keep(sc, s["mod"], sh.cu, s["counts"], case["mode"] == "joint")
        return dict(scores=sc, keep=kept.int(), modality=s["mod"][kept], k=s["k"][:, kept], v=s["v"][:, kept],
                    hidden=s["h"][kept], cu=new.cpu().numpy().astype(np.int32))
    if kind == "schedule":
        sh, pp, layers = s["shape"], s["pp"], s["layers"]
        rows = torch.arange(sh.T, device="cuda")
        cu, keeps, cus, before = sh.cu, [], [], None
        mod = pp.modality_in
        for i, l in enumerate(layers):
            sc = _exact_scores(pp.q[i], pp.k_in[l - layers[0]][rows], mod[rows], cu, sh.cuq, case["domain"] == "causal")
            kept, new = _exact_keep(sc, mod[rows], cu, s["counts"][i], case["mode"] == "joint")
            keeps.append(kept.int())
            cu = new.cpu().numpy().astype(np.int32)
            cus.append(cu)
            before, rows = rows, rows[kept]
        top, prev = layers[-1] - layers[0], layers[-2] - layers[0]
        return dict(scores=sc, keep=keeps, modality=mod[rows], k=pp.k_in[top:, rows], v=pp.v_in[top:, rows],
                    k_before=pp.k_in[prev:, before], v_before=pp.v_in[prev:, before], hidden=pp.hidden_in[rows], cu=cus)
    if kind == "decode":
        hq, hkv = _heads(case)
        out = torch.zeros(s["q"].shape, dtype=torch.float64, device="cuda")
        for b in range(case["seqs"]):
            t = slice(int(s["cu"][b]), int(s["cu"][b + 1]))
            q = s["q"][b].double().view(hkv, hq // hkv, D)
            k, v = s["k"][t].double().transpose(0, 1), s["v"][t].double().transpose(0, 1)
            out[b] = (torch.softmax(q @ k.transpose(1, 2) / math.sqrt(D), -1) @ v).reshape(hq, D)
        return out
    return _exact_align(s)


def _exact_align(s, tau=0.78, beta=0.90):
    case = s["case"]
    F, tpf, dim, W, n = case["frames"], case["tpf"], case["dim"], case["window"], s["n_audio"]
    v = s["visual"].view(F, tpf, dim).sum(1, dtype=torch.float64) / tpf
    at = (torch.arange(n, device="cuda") * F) // n
    a = torch.zeros(F, dim, dtype=torch.float64, device="cuda").index_add_(0, at, s["audio"].double())
    a /= torch.bincount(at, minlength=F)[:, None]
    c = torch.zeros(F, dtype=torch.float64, device="cuda")
    for f in range(F):
        w = slice(max(0, f - W // 2), min(F, f + W // 2 + 1))
        ka, kv = a[w] - a[w].mean(0), v[w] - v[w].mean(0)
        ka, kv = ka @ ka.T, kv @ kv.T
        den = ka.norm() * kv.norm()
        c[f] = torch.where(den > 0, (ka * kv).sum() / den, torch.zeros_like(den))
    d = (v - a).norm(dim=1)
    dn = (d - d.min()) / (d.max() - d.min())
    cbar = c.mean()
    score = (1 - beta) * c + beta * (1 - dn) if float(cbar) < tau else c
    return dict(c=c, s=score, dnorm=dn, cbar=cbar.view(1))
