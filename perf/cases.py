"""The calls of the AVTP pruning stage whose time is followed.

Three kinds of call make up the work of a program that uses this library:

* ``prune``: the whole pruning stage at a decoder layer (score, allocate, select, compact),
  by hidden-state variation (the default criterion) or by text attention;
* ``score``: the text-attention criterion alone, with its own normaliser, with one kept by
  the layer's attention, or for the request's last token as the only query;
* ``forward``: the pruning layer's causal attention, with the text-attention scores as its
  side output.

A case is a layout (requests of images and text, drawn from the case's own numbers) and the
shape of the model's tensors. The values come from the seed: normal hidden states, queries,
keys and values, with an importance of its own for every image. Every pass runs a prepared
call on buffers that a serving program would keep for its layout.
"""
from __future__ import annotations

import math
import random
from typing import Dict, List

import numpy as np
import torch

from paper_2608_26806_gb300 import avtp

DEV = "cuda"

# hidden, query heads, KV heads, head_dim, position-id planes of the models' layers
TINY = dict(hidden=256, q_heads=4, kv_heads=2, head_dim=64, planes=1)
LLAVA = dict(hidden=3584, q_heads=28, kv_heads=4, head_dim=128, planes=1)
QWEN = dict(hidden=4096, q_heads=32, kv_heads=8, head_dim=128, planes=3)
INTERN = dict(hidden=4096, q_heads=32, kv_heads=8, head_dim=128, planes=1)

# a layout: per request, `lead` text tokens, then images of image_min..image_max tokens (a
# multiple of image_step), each behind `gap` text tokens, then the rest of its text
TINY_REQUEST = dict(layout=1, requests=1, images_min=3, images_max=3, image_min=64, image_max=64, image_step=1,
                    lead=0, gap=0, text_min=32, text_max=32, keep=0.5)
LLAVA_REQUEST = dict(layout=1, requests=1, images_min=8, images_max=8, image_min=729, image_max=729, image_step=1,
                     lead=0, gap=8, text_min=128, text_max=128, keep=0.25)
QWEN_REQUEST = dict(layout=3, requests=1, images_min=16, images_max=16, image_min=256, image_max=1024, image_step=64,
                    lead=64, gap=2, text_min=256, text_max=256, keep=0.33)
SERVING_BATCH = dict(layout=4, requests=8, images_min=4, images_max=32, image_min=256, image_max=256, image_step=1,
                     lead=0, gap=2, text_min=64, text_max=512, keep=0.33)
LONG_BATCH = dict(layout=5, requests=4, images_min=64, images_max=64, image_min=1024, image_max=1024, image_step=1,
                  lead=0, gap=2, text_min=512, text_max=512, keep=0.125)


def listed() -> List[Dict]:
    def case(name, op, how, shape, layout):
        return dict(name=name, op=op, how=how, **shape, **layout)

    return [
        # the smallest stage a program runs: three small images; launches and latency are all of it
        case("prune_tiny", "prune", "hidden", TINY, TINY_REQUEST),
        # one chat request of eight fixed-size images: an odd token count and a hidden size of 28 * 128
        case("prune_llava", "prune", "hidden", LLAVA, LLAVA_REQUEST),
        # one chat request of sixteen images of mixed resolution, three planes of position ids
        case("prune_qwen", "prune", "hidden", QWEN, QWEN_REQUEST),
        # a serving batch of eight ragged requests
        case("prune_serving", "prune", "hidden", INTERN, SERVING_BATCH),
        # the largest: four requests of 64 large images each (video frames), 264 thousand tokens
        case("prune_long", "prune", "hidden", INTERN, LONG_BATCH),
        # the serving batch pruned by what its text attends to
        case("prune_text_serving", "prune", "text", INTERN, SERVING_BATCH),
        # text attention of one request, with its own normaliser: the layer statistic's inner call
        case("score_text_qwen", "score", "text", QWEN, QWEN_REQUEST),
        # the same criterion where the layer's attention kept its normaliser; seven heads a group
        case("score_lse_llava", "score", "lse", LLAVA, LLAVA_REQUEST),
        # the attention of the token that predicts the first generated one
        case("score_last_qwen", "score", "last", QWEN, QWEN_REQUEST),
        # the pruning layer's attention in a prefill, with the scores it gives: one request each
        # of the two models, and the serving batch
        case("forward_llava", "forward", "text", LLAVA, LLAVA_REQUEST),
        case("forward_qwen", "forward", "text", QWEN, QWEN_REQUEST),
        case("forward_serving", "forward", "text", INTERN, SERVING_BATCH),
    ]


def draw(rng: random.Random) -> Dict:
    op, how, most = rng.choice([("prune", "hidden", 262144), ("prune", "hidden", 262144), ("prune", "text", 65536),
                                ("score", "text", 65536), ("score", "lse", 65536), ("score", "last", 65536),
                                ("forward", "text", 32768), ("forward", "plain", 32768)])

    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    # pruned by text attention: a serving batch of tiles, where one near-tie moves few of the kept rows
    tiles = (op, how) == ("prune", "text")
    tokens = log_uniform(16384 if tiles else 224, most)
    requests = min(rng.choice([1, 1, 1, 2, 3, 4, 6, 8]), max(1, tokens // 200))
    if op == "forward":  # no request longer than the serving batch's: the work grows with the square
        requests = max(requests, -(-tokens // 8192))
    share = tokens // requests
    image_max = min(log_uniform(32, 256 if tiles else 1024), share)
    image_min = rng.randint(max(1, image_max // 4), image_max)
    images = max(1, min(256 if tiles else 64, round(share / ((image_min + image_max) / 2))))
    gap = rng.choice([0, 1, 2, 8])
    lead = rng.choice([0, 8, 64])
    text_min = lead + gap * images + rng.randint(1, 64)
    shape = rng.choice([TINY, LLAVA, QWEN, INTERN])
    return dict(op=op, how=how, **shape, layout=rng.randrange(1 << 30), requests=requests,
                images_min=max(1, images - images // 4), images_max=images, image_min=image_min, image_max=image_max,
                image_step=1, lead=lead, gap=gap, text_min=text_min, text_max=text_min + rng.choice([0, 7, 128]),
                keep=rng.choice([0.125, 0.25, 0.33, 0.5]))


# ---------------------------------------------------------------- layout
def layout_of(case: Dict) -> Dict[str, np.ndarray]:
    rng = random.Random(case["layout"])
    cu, img_cu, start, length = [0], [0], [], []
    for _ in range(case["requests"]):
        m = rng.randint(case["images_min"], case["images_max"])
        steps = (case["image_max"] - case["image_min"]) // case["image_step"]
        sizes = [case["image_min"] + case["image_step"] * rng.randint(0, steps) for _ in range(m)]
        text = rng.randint(case["text_min"], case["text_max"])
        gap = min(case["gap"], max(0, text - case["lead"] - 1) // m)
        pos = min(case["lead"], text - 1)
        rest = text - pos - gap * m
        for n in sizes:
            pos += gap
            start.append(pos)
            length.append(n)
            pos += n
        cu.append(cu[-1] + pos + rest)
        img_cu.append(len(length))
    return {k: np.asarray(v, dtype=np.int32) for k, v in dict(cu_seqlens=cu, img_cu=img_cu, img_start=start,
                                                              img_len=length).items()}


def rows_of(lay: Dict[str, np.ndarray]):
    """Per packed token: its request, and its image or -1 (int64 arrays)."""
    T, R = int(lay["cu_seqlens"][-1]), len(lay["cu_seqlens"]) - 1
    req = np.repeat(np.arange(R), np.diff(lay["cu_seqlens"]))
    img = np.full(T, -1, dtype=np.int64)
    for r in range(R):
        for i in range(lay["img_cu"][r], lay["img_cu"][r + 1]):
            a = int(lay["cu_seqlens"][r]) + int(lay["img_start"][i])
            img[a:a + int(lay["img_len"][i])] = i
    return req, img


# ---------------------------------------------------------------- inputs
def hidden_states(case, gen, img, signal):
    """h_prior = N(0,1) and h_cur = h_prior + beta N(0,1), beta = 0.25 + the image's signal."""
    T, D = len(img), case["hidden"]
    beta = torch.full((T, 1), 0.25, device=DEV)
    vis = img >= 0
    beta[vis, 0] += signal[img[vis]]
    prior = torch.randn(T, D, device=DEV, dtype=torch.bfloat16, generator=gen)
    cur = torch.empty_like(prior)
    for a in range(0, T, 32768):
        b = min(T, a + 32768)
        cur[a:b] = prior[a:b] + beta[a:b] * torch.randn(b - a, D, device=DEV, generator=gen)
    return cur, prior


def heads(case, gen, req, img, signal, R):
    """q, k and v = N(0,1), the keys of an image moved towards its request's mean text query."""
    T, Hq, Hkv, d = len(img), case["q_heads"], case["kv_heads"], case["head_dim"]
    q = torch.randn(T, Hq, d, device=DEV, dtype=torch.bfloat16, generator=gen)
    mean = torch.zeros(R, Hkv, d, device=DEV)
    for r in range(R):
        rows = torch.nonzero((req == r) & (img < 0)).flatten()
        if rows.numel():
            mean[r] = q[rows].float().view(-1, Hkv, Hq // Hkv, d).mean((0, 2))
    row = torch.where(img >= 0, signal[img.clamp(min=0)], torch.zeros((), device=DEV))
    k = torch.empty(T, Hkv, d, device=DEV, dtype=torch.bfloat16)
    for a in range(0, T, 32768):
        n = min(T, a + 32768) - a
        k[a:a + n] = (torch.randn(n, Hkv, d, device=DEV, generator=gen)
                      + row[a:a + n, None, None] * mean[req[a:a + n]])
    v = torch.randn(T, Hkv, d, device=DEV, dtype=torch.bfloat16, generator=gen)
    return q, k, v


def inputs(case: Dict, seed: int):
    lay = layout_of(case)
    req, img = (torch.from_numpy(x).to(DEV) for x in rows_of(lay))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    NI, R = len(lay["img_len"]), case["requests"]
    # a few images matter much, most a little
    signal = torch.exp(torch.randn(NI, device=DEV, generator=gen))
    signal = signal / signal.max().clamp(min=1e-6)
    got = {}
    if case["op"] == "prune":
        T = len(img)
        got["pos"] = (torch.arange(T, device=DEV, dtype=torch.int32)[None]
                      + T * torch.arange(case["planes"], device=DEV, dtype=torch.int32)[:, None]).contiguous()
        got["h_cur"], got["h_prior"] = hidden_states(case, gen, img, signal)
        if case["how"] != "hidden":
            del got["h_prior"]
    if case["how"] != "hidden":
        got["q"], got["k"], got["v"] = heads(case, gen, req, img, signal, R)
        if case["op"] != "forward":
            del got["v"]
    if case["how"] == "lse":  # what the layer's attention would have kept, from plain 32-bit products
        got["lse"] = torch.zeros(case["q_heads"], len(img), device=DEV)
        for pos, z in text_logits(lay, got["q"], got["k"], torch.float32):
            got["lse"][:, pos] = torch.logsumexp(z, dim=2)
    return lay, got


def text_logits(lay, q, k, dtype, last=False, most=1 << 27):
    """(positions, scaled causal logits [Hq, positions, tokens up to the last of them]) of the text
    queries of every request, a chunk of queries at a time; `last`: of its last token alone."""
    _, img = rows_of(lay)
    G = q.shape[1] // k.shape[1]
    for a, b in zip(lay["cu_seqlens"][:-1], lay["cu_seqlens"][1:]):
        a, b = int(a), int(b)
        where = np.asarray([b - 1]) if last else a + np.nonzero(img[a:b] < 0)[0]
        step = max(1, most // (q.shape[1] * (b - a)))
        for c in range(0, len(where), step):
            pos = torch.from_numpy(where[c:c + step]).to(DEV)
            end = int(where[min(len(where), c + step) - 1]) + 1
            kk = k[a:end].to(dtype).permute(1, 2, 0)
            qq = q[pos].to(dtype).permute(1, 0, 2).reshape(k.shape[1], G * len(pos), -1)
            z = torch.matmul(qq, kk).view(q.shape[1], len(pos), end - a) * (q.shape[2] ** -0.5)
            hidden = torch.arange(a, end, device=DEV)[None, :] > pos[:, None]
            yield pos, z.masked_fill_(hidden[None], -math.inf)


def prepare(case: Dict, seed: int):
    lay, x = inputs(case, seed)
    L = avtp.Layout.from_host(**lay, device=DEV)
    state = dict(case=case, layout=L, inputs=x)
    if case["op"] == "prune":
        keep = np.full(case["requests"], case["keep"], dtype=np.float32)
        tensors = dict(h_cur=x["h_cur"], h_prior=x["h_prior"]) if case["how"] == "hidden" else dict(q=x["q"], k=x["k"])
        state["call"] = avtp.PruneCall(L, "hidden_variation" if case["how"] == "hidden" else "text_attention",
                                       keep_ratio=torch.from_numpy(keep).to(DEV), keep_ratio_host=keep,
                                       rows={"hidden": x["h_cur"]}, planes={"pos": x["pos"]}, **tensors)
    elif case["op"] == "score":
        args = dict(q=x["q"], k=x["k"], lse=x.get("lse"), query_set="last" if case["how"] == "last" else "text")
        state["args"] = dict(args, scores=torch.zeros(L.n_tokens, device=DEV),
                             img_sums=torch.empty(L.n_images, dtype=torch.int64, device=DEV),
                             workspace=avtp.new_workspace(avtp.workspace_size(L, "text_attention", **args), DEV))
    else:
        state["call"] = avtp.ForwardCall(L, q=x["q"], k=x["k"], v=x["v"], scores=case["how"] == "text")
    return state


def run(state):
    op = state["case"]["op"]
    if op == "prune":
        b = state["call"].run()
        # the kept rows are copies: compared bit for bit, as whole numbers
        return dict(scores=b.scores, budgets=b.budgets, offsets=b.out_cu_seqlens, kept=b.kept_idx,
                    hidden=b.outputs["hidden"].view(torch.int16), pos=b.outputs["pos"])
    if op == "score":
        scores, sums = avtp.score(state["layout"], "text_attention", **state["args"])
        return dict(scores=scores, sums=sums.double())  # fixed point, 2^-32: compared as numbers
    c = state["call"].run()
    return dict(o=c.o, lse=c.lse) if c.scores is None else dict(o=c.o, lse=c.lse, scores=c.scores)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case: Dict) -> Dict[str, float]:
    lay = layout_of(case)
    req, img = rows_of(lay)
    T, vis = len(img), int((img >= 0).sum())
    R, D, P = case["requests"], case["hidden"], case["planes"]
    Hq, Hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    counts = np.bincount(req[img >= 0], minlength=R)
    text = np.bincount(req[img < 0], minlength=R)
    kept = int(sum(math.floor(np.float64(np.float32(case["keep"])) * n + 0.5) for n in counts)) + T - vis
    nbytes = flops = 0.0
    # text attention: every logit of a query and a key it sees, once, from each key and query read once
    pos = np.arange(T) - lay["cu_seqlens"][req] + 1
    if case["how"] in ("text", "lse") and case["op"] != "forward":
        nbytes += 2.0 * d * (Hkv * T + Hq * int(text.sum())) + 4.0 * vis
        pairs = pos[img < 0].sum()
        if case["how"] == "lse":  # the visual keys alone
            before = np.concatenate([[0], np.cumsum(img >= 0)])
            pairs = sum(before[t + 1] - before[lay["cu_seqlens"][req[t]]] for t in np.nonzero(img < 0)[0])
            nbytes += 4.0 * Hq * int(text.sum()) - 2.0 * d * Hkv * (T - vis)
        flops += 2.0 * d * Hq * float(pairs)
    if case["how"] == "last":
        nbytes += 2.0 * d * (Hkv * T + Hq * R) + 4.0 * vis
        flops += 2.0 * d * Hq * T
    if case["op"] == "prune":
        if case["how"] == "hidden":  # both rows of every visual token, the current row of every text token
            nbytes += 2.0 * D * (2 * vis + (T - vis)) + 4.0 * vis
            flops += 6.0 * D * vis
        else:  # the kept rows alone
            nbytes += 2.0 * D * kept
        nbytes += 2.0 * D * kept + 8.0 * P * kept + 4.0 * kept
    if case["op"] == "forward":
        nbytes += 2.0 * d * T * (Hq + 2 * Hkv) + 4.0 * T * Hq * (d + 1) + (4.0 * vis if case["how"] == "text" else 0.0)
        flops += 4.0 * d * Hq * float(pos.sum())
    return dict(bytes=nbytes, flops=flops)


def tolerance(case: Dict):
    if case["op"] == "forward":
        # the probabilities are rounded to bf16 before their product with the values: O is 1.3e-3
        # (2-norm) from `exact`, the normaliser and the scores are 1e-7
        return {"rel": 5e-3}
    # 32-bit sums over a hidden row, or over a key's queries and heads: 2e-7 to 8e-7 from `exact`.
    # Whole numbers: a near-tie that falls the other way moves the kept rows of one image.
    return {"rel": 4e-6, "max": 2e-4, "differ": 0.01} if case["op"] == "prune" else {"rel": 4e-6, "max": 2e-4}


# ---------------------------------------------------------------- the same in 64 bits
def exact(case: Dict, seed: int):
    lay, x = inputs(case, seed)
    req, img = rows_of(lay)
    vis = torch.from_numpy(np.nonzero(img >= 0)[0]).to(DEV)
    scores = torch.zeros(len(img), dtype=torch.float64, device=DEV)
    if case["how"] == "hidden":
        for a in range(0, len(vis), 16384):
            t = vis[a:a + 16384]
            c, p = x["h_cur"][t].double(), x["h_prior"][t].double()
            dot, cc, pp = (c * p).sum(1), c.square().sum(1).sqrt(), p.square().sum(1).sqrt()
            scores[t] = 1 - dot / (cc.clamp(min=1e-8) * pp.clamp(min=1e-8))
    elif case["how"] != "plain":
        queries = np.ones(case["requests"]) if case["how"] == "last" else np.bincount(req[img < 0],
                                                                                      minlength=case["requests"])
        for pos, z in text_logits(lay, x["q"], x["k"], torch.float64, last=case["how"] == "last"):
            r = int(req[int(pos[0])])
            a = int(lay["cu_seqlens"][r])
            norm = x["lse"][:, pos].double()[:, :, None] if case["how"] == "lse" else torch.logsumexp(z, 2, True)
            scores[a:a + z.shape[2]] += torch.exp(z - norm).sum((0, 1)) / (case["q_heads"] * float(queries[r]))
        scores *= torch.from_numpy((img >= 0).astype(np.float64)).to(DEV)
    if case["op"] == "prune":
        return dict(scores=scores, budgets=None, offsets=None, kept=None, hidden=None, pos=None)
    if case["op"] == "score":
        sums = torch.zeros(len(lay["img_len"]), dtype=torch.float64, device=DEV)
        sums.index_add_(0, torch.from_numpy(img).to(DEV)[vis], scores[vis])
        return dict(scores=scores, sums=sums * 2.0 ** 32)
    q, k, v = x["q"], x["k"], x["v"]
    Hq, Hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    G = Hq // Hkv
    o = torch.empty(len(img), Hq, d, dtype=torch.float64, device=DEV)
    lse = torch.empty(Hq, len(img), dtype=torch.float64, device=DEV)
    for a, b in zip(lay["cu_seqlens"][:-1], lay["cu_seqlens"][1:]):
        a, b = int(a), int(b)
        for c in range(a, b, 512):
            e = min(b, c + 512)
            kk, vv = k[a:e].double().transpose(0, 1), v[a:e].double().transpose(0, 1)
            qq = q[c:e].double().permute(1, 0, 2).reshape(Hkv, G * (e - c), d)
            z = torch.matmul(qq, kk.transpose(1, 2)).view(Hkv, G, e - c, e - a) * (d ** -0.5)
            hidden = torch.arange(a, e, device=DEV)[None, :] > torch.arange(c, e, device=DEV)[:, None]
            z.masked_fill_(hidden, -math.inf)
            n = torch.logsumexp(z, dim=3)
            p = torch.exp(z - n[..., None]).view(Hkv, G * (e - c), e - a)
            o[c:e] = torch.matmul(p, vv).view(Hq, e - c, d).transpose(0, 1)
            lse[:, c:e] = n.reshape(Hq, e - c)
    return dict(o=o, lse=lse) if case["how"] == "plain" else dict(o=o, lse=lse, scores=scores)
