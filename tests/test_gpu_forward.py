"""GPU parity of the layer's causal attention forward (avtp_attn_forward) and of the
text-attention scores it produces from its own LSE, against the fp64 oracle.

Tolerances, from the arithmetic:
- LSE: rel 1e-3 / abs 1e-5. The kernel sums fp32 exponentials of fp32 logits of bf16
  inputs, so its error is near fp32 rounding.
- O: |O - O_ref| <= 2^-8 * O_abs + 1e-5 element by element, where O_abs is the forward
  of |v|. The kernel rounds each probability p to bf16 before P V (as FlashAttention
  does), and bf16 rounding moves p by at most 2^-8 p, so the weighted sum moves by at
  most 2^-8 sum p |v| / l. The rounding errors are of both signs, so their mean over
  all elements must also stay below 2^-10 * O_abs.
- Scores: rel 1e-3 / abs 1e-5, as for avtp_score; image sums exact for the GPU's
  own scores.
"""
import numpy as np
import pytest
import torch

from oracle import avtp_oracle as O
from paper_2608_26806_gb300 import avtp, synth
from tests.gpu_util import ATOL, RTOL, assert_scores_close, bf16_dev, dev_layout, ensure_built

pytestmark = pytest.mark.gpu

O_REL = 2.0 ** -8
O_MEAN_REL = 2.0 ** -10


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_built()


def _dev(wl):
    L = dev_layout(wl.layout)
    return L, bf16_dev(wl.q), bf16_dev(wl.k), bf16_dev(wl.v)


def _check_o(got, ref, ref_abs):
    err = np.abs(got - ref)
    bound = O_REL * ref_abs + 1e-5
    worst = np.argmax(err - bound)
    assert np.all(err <= bound), (f"O outside its bound at {np.unravel_index(worst, err.shape)}: "
                                  f"{got.flat[worst]} vs {ref.flat[worst]} (bound {bound.flat[worst]})")
    assert err.sum() <= O_MEAN_REL * ref_abs.sum() + 1e-7 * err.size


def _abs_v(v_bits):
    return (v_bits & np.uint16(0x7FFF)).astype(np.uint16)


# Layouts for the forward: requests of 1, 127, 128, 129 and several hundred tokens that
# start at packed offsets that are not multiples of 128 (so query tiles and key blocks
# straddle request boundaries), text only, images only, and many query tiles.
_FWD_LAYOUTS = [
    [[("t", 1)]],
    [[("i", 64), ("t", 63)], [("t", 1), ("i", 127), ("t", 1)], [("i", 200), ("t", 57)], [("t", 128)]],
    [[("t", 5), ("i", 300), ("t", 3)], [("i", 128)], [("t", 130), ("i", 385), ("t", 2)]],
    [[("t", 70), ("i", 129), ("i", 1), ("t", 1)], [("i", 40), ("t", 3), ("i", 600), ("t", 100)]],
]


@pytest.mark.parametrize("layout_id", range(len(_FWD_LAYOUTS)))
@pytest.mark.parametrize("heads", [(4, 4, 64), (6, 2, 64), (12, 4, 128), (7, 1, 128)])
def test_forward_matches_oracle(layout_id, heads):
    Hq, Hkv, d = heads
    wl = synth.make_custom(_FWD_LAYOUTS[layout_id], n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, hidden=64,
                           seed=31 + layout_id, parts=("B", "V"))
    L, q, k, v = _dev(wl)
    o, lse, scores, sums = avtp.attn_forward(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale)
    torch.cuda.synchronize()
    ref_o, ref_lse = O.attention_forward(wl.layout, wl.q, wl.k, wl.v, Hq, Hkv, wl.softmax_scale)
    ref_abs, _ = O.attention_forward(wl.layout, wl.q, wl.k, _abs_v(wl.v), Hq, Hkv, wl.softmax_scale)
    _check_o(o.cpu().numpy(), ref_o, ref_abs)
    np.testing.assert_allclose(lse.cpu().numpy(), ref_lse, rtol=RTOL, atol=ATOL)
    # criterion B from the forward's LSE
    got = scores.cpu().numpy()
    vis = wl.layout.visual_mask()
    if vis.any():
        ref = O.score_text_attention(wl.layout, wl.q, wl.k, Hq, Hkv, wl.softmax_scale)
        assert_scores_close(got, ref, vis)
        assert np.array_equal(sums.cpu().numpy(), O.image_sums(wl.layout, got))


@pytest.mark.parametrize("query_set,path", [("text", "tensor"), ("text", "cuda"), ("last", "auto")])
def test_forward_side_output_on_each_scoring_path(query_set, path):
    wl = synth.make_custom(_FWD_LAYOUTS[2], n_q_heads=8, n_kv_heads=2, head_dim=128, hidden=64, seed=5,
                           parts=("B", "V"))
    L, q, k, v = _dev(wl)
    _, lse, scores, sums = avtp.attn_forward(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale, query_set=query_set,
                                             path=path)
    torch.cuda.synchronize()
    got = scores.cpu().numpy()
    ref = O.score_text_attention(wl.layout, wl.q, wl.k, 8, 2, wl.softmax_scale, query_set=query_set)
    assert_scores_close(got, ref, wl.layout.visual_mask())
    assert np.array_equal(sums.cpu().numpy(), O.image_sums(wl.layout, got))


def test_plain_forward_leaves_scores_alone():
    wl = synth.make_custom(_FWD_LAYOUTS[1], n_q_heads=4, n_kv_heads=2, head_dim=64, hidden=64, seed=9,
                           parts=("B", "V"))
    L, q, k, v = _dev(wl)
    o, lse, scores, sums = avtp.attn_forward(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale, scores=False)
    torch.cuda.synchronize()
    assert scores is None and sums is None
    ref_o, ref_lse = O.attention_forward(wl.layout, wl.q, wl.k, wl.v, 4, 2, wl.softmax_scale)
    ref_abs, _ = O.attention_forward(wl.layout, wl.q, wl.k, _abs_v(wl.v), 4, 2, wl.softmax_scale)
    _check_o(o.cpu().numpy(), ref_o, ref_abs)
    np.testing.assert_allclose(lse.cpu().numpy(), ref_lse, rtol=RTOL, atol=ATOL)


def test_forward_repeatable():
    wl = synth.make_custom(_FWD_LAYOUTS[3], n_q_heads=6, n_kv_heads=2, head_dim=128, hidden=64, seed=3,
                           parts=("B", "V"))
    L, q, k, v = _dev(wl)
    c = avtp.ForwardCall(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale)
    c.run()
    o1, l1, s1 = c.o.clone(), c.lse.clone(), c.scores.clone()
    c.run()
    torch.cuda.synchronize()
    assert torch.equal(o1, c.o) and torch.equal(l1, c.lse) and torch.equal(s1, c.scores)
    assert avtp.read_device_status(c.workspace) == 0


# ---------------------------------------------------------------- full-size workloads
@pytest.mark.parametrize("name", ["qwen3_vl_8b", "llava_ov_7b"])
def test_forward_full_size_sampled_rows(name):
    """The workload the bench times: O and the LSE of sampled rows (the first and last rows
    of query tiles, the request's last token) against the oracle's per-row forward, the
    LSE of every text query against the oracle's, and the scores in full."""
    wl = synth.make_workload(name, parts=("B", "V"))
    L, q, k, v = _dev(wl)
    Hq, Hkv = wl.n_q_heads, wl.n_kv_heads
    o, lse, scores, sums = avtp.attn_forward(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale)
    torch.cuda.synchronize()
    T = wl.layout.n_tokens
    rows = sorted({0, 1, 127, 128, 129, 2047, 2048, T // 2, T - 129, T - 128, T - 2, T - 1})
    ref_o, ref_lse = O.attention_forward_rows(wl.layout, wl.q, wl.k, wl.v, Hq, Hkv, wl.softmax_scale, 0, rows)
    ref_abs, _ = O.attention_forward_rows(wl.layout, wl.q, wl.k, _abs_v(wl.v), Hq, Hkv, wl.softmax_scale, 0, rows)
    _check_o(o[rows].cpu().numpy(), ref_o, ref_abs)
    np.testing.assert_allclose(lse[:, rows].cpu().numpy(), ref_lse, rtol=RTOL, atol=ATOL)
    text = ~wl.layout.visual_mask()
    ref_text_lse = O.text_lse(wl.layout, wl.q, wl.k, Hq, Hkv, wl.softmax_scale)
    np.testing.assert_allclose(lse.cpu().numpy()[:, text], ref_text_lse[:, text], rtol=RTOL, atol=ATOL)
    got = scores.cpu().numpy()
    ref = O.score_text_attention(wl.layout, wl.q, wl.k, Hq, Hkv, wl.softmax_scale)
    assert_scores_close(got, ref, wl.layout.visual_mask())
    assert np.array_equal(sums.cpu().numpy(), O.image_sums(wl.layout, got))


def test_forward_serving_batch_sampled_rows():
    """Eight varlen requests: sampled rows of every request (its first, tile-edge and last
    tokens) against the oracle."""
    wl = synth.make_workload("internvl3_5_8b", parts=("B", "V"))
    L, q, k, v = _dev(wl)
    Hq, Hkv = wl.n_q_heads, wl.n_kv_heads
    o, lse, _, _ = avtp.attn_forward(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale, scores=False)
    torch.cuda.synchronize()
    cu = wl.layout.cu_seqlens
    o_h, lse_h = o.cpu().numpy(), lse.cpu().numpy()
    for r in range(wl.layout.n_requests):
        n = int(cu[r + 1] - cu[r])
        rows = sorted({0, 127, 128, n // 2, n - 1})
        ref_o, ref_lse = O.attention_forward_rows(wl.layout, wl.q, wl.k, wl.v, Hq, Hkv, wl.softmax_scale, r, rows)
        ref_abs, _ = O.attention_forward_rows(wl.layout, wl.q, wl.k, _abs_v(wl.v), Hq, Hkv, wl.softmax_scale, r,
                                              rows)
        g = [int(cu[r]) + p for p in rows]
        _check_o(o_h[g], ref_o, ref_abs)
        np.testing.assert_allclose(lse_h[:, g], ref_lse, rtol=RTOL, atol=ATOL)


def test_forward_many_small_requests():
    """Forty requests of 1 to 300 tokens: many query tiles per call, tiles and key blocks
    that straddle request boundaries at every offset, requests shorter than a tile."""
    rng = np.random.default_rng(17)
    reqs = []
    for _ in range(40):
        segs = []
        for _ in range(int(rng.integers(1, 4))):
            segs.append(("t" if rng.random() < 0.5 else "i", int(rng.integers(1, 101))))
        reqs.append(segs)
    wl = synth.make_custom(reqs, n_q_heads=4, n_kv_heads=1, head_dim=64, hidden=64, seed=23, parts=("B", "V"))
    L, q, k, v = _dev(wl)
    o, lse, scores, sums = avtp.attn_forward(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale)
    torch.cuda.synchronize()
    ref_o, ref_lse = O.attention_forward(wl.layout, wl.q, wl.k, wl.v, 4, 1, wl.softmax_scale)
    ref_abs, _ = O.attention_forward(wl.layout, wl.q, wl.k, _abs_v(wl.v), 4, 1, wl.softmax_scale)
    _check_o(o.cpu().numpy(), ref_o, ref_abs)
    np.testing.assert_allclose(lse.cpu().numpy(), ref_lse, rtol=RTOL, atol=ATOL)
    vis = wl.layout.visual_mask()
    ref = O.score_text_attention(wl.layout, wl.q, wl.k, 4, 1, wl.softmax_scale)
    assert_scores_close(scores.cpu().numpy(), ref, vis)


def test_forward_strided_tensors():
    """q, k and v rows with padded token strides, O and the LSE written into wider buffers:
    the strides of the ABI are honoured and nothing outside the views is written."""
    Hq, Hkv, d = 6, 2, 128
    wl = synth.make_custom(_FWD_LAYOUTS[2], n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, hidden=64, seed=41,
                           parts=("B", "V"))
    T = wl.layout.n_tokens
    L = dev_layout(wl.layout)

    def padded(bits, heads):
        big = torch.zeros(T, heads + 1, d, dtype=torch.bfloat16, device="cuda")
        big[:, :heads] = bf16_dev(bits)
        return big[:, :heads]

    q, k, v = padded(wl.q, Hq), padded(wl.k, Hkv), padded(wl.v, Hkv)
    o_big = torch.full((T, Hq + 2, d), 7.0, dtype=torch.float32, device="cuda")
    lse_big = torch.full((Hq, T + 24), 7.0, dtype=torch.float32, device="cuda")
    c = avtp.ForwardCall(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale, o=o_big[:, :Hq], lse=lse_big[:, :T])
    c.run()
    torch.cuda.synchronize()
    ref_o, ref_lse = O.attention_forward(wl.layout, wl.q, wl.k, wl.v, Hq, Hkv, wl.softmax_scale)
    ref_abs, _ = O.attention_forward(wl.layout, wl.q, wl.k, _abs_v(wl.v), Hq, Hkv, wl.softmax_scale)
    _check_o(o_big[:, :Hq].cpu().numpy(), ref_o, ref_abs)
    np.testing.assert_allclose(lse_big[:, :T].cpu().numpy(), ref_lse, rtol=RTOL, atol=ATOL)
    assert torch.all(o_big[:, Hq:] == 7.0) and torch.all(lse_big[:, T:] == 7.0)
    ref = O.score_text_attention(wl.layout, wl.q, wl.k, Hq, Hkv, wl.softmax_scale)
    assert_scores_close(c.scores.cpu().numpy(), ref, wl.layout.visual_mask())


# ---------------------------------------------------------------- the softmax's reference, tile edges
# A row's reference moves when a half block's sum of exponentials leaves its range: keys that
# grow along the sequence move it again and again, in first and second halves of a block.
@pytest.mark.parametrize("heads", [(4, 2, 64), (3, 1, 64), (8, 2, 128), (3, 3, 128)])
@pytest.mark.parametrize("growth", [40.0, -40.0, 400.0])
def test_forward_moving_reference(heads, growth):
    Hq, Hkv, d = heads
    wl = synth.make_custom([[("t", 3), ("i", 500), ("t", 27)], [("i", 64), ("t", 129)]], n_q_heads=Hq, n_kv_heads=Hkv,
                           head_dim=d, hidden=64, seed=77, parts=("B", "V"))
    T = wl.layout.n_tokens
    rng = np.random.default_rng(5)
    # logits that climb (or fall) by `growth` over 500 keys, in steps of their own size, the
    # same for every query: q = 1 / d everywhere plus noise, k = ramp + noise
    ramp = growth * (np.arange(T) // 37) * 37 / 500.0
    scale = 1.0
    q = (np.full((T, Hq, d), 1.0 / d) + 0.002 * rng.standard_normal((T, Hq, d))).astype(np.float32)
    k = (ramp[:, None, None] + rng.standard_normal((T, Hkv, d))).astype(np.float32)
    wl.tensors["q"] = synth.f32_to_bf16_bits(q.reshape(T, -1)).reshape(T, Hq, d)
    wl.tensors["k"] = synth.f32_to_bf16_bits(k.reshape(T, -1)).reshape(T, Hkv, d)
    L, qd, kd, vd = _dev(wl)
    o, lse, _, _ = avtp.attn_forward(L, q=qd, k=kd, v=vd, softmax_scale=scale, scores=False)
    torch.cuda.synchronize()
    ref_o, ref_lse = O.attention_forward(wl.layout, wl.q, wl.k, wl.v, Hq, Hkv, scale)
    ref_abs, _ = O.attention_forward(wl.layout, wl.q, wl.k, _abs_v(wl.v), Hq, Hkv, scale)
    # fp32 logits of up to 440 (products of up to 7): their sum is off by at most d 2^-24 times
    # sum |q k| = 128 * 2^-24 * 500 < 4e-3, which moves a probability by as much of itself
    err = np.abs(o.cpu().numpy() - ref_o)
    assert np.all(err <= (O_REL + (4e-3 if growth == 400.0 else 4e-4)) * ref_abs + 1e-5)
    np.testing.assert_allclose(lse.cpu().numpy(), ref_lse, rtol=RTOL, atol=4e-3 if growth == 400.0 else 4e-4)


@pytest.mark.parametrize("heads", [(4, 2, 64), (3, 1, 128)])
@pytest.mark.parametrize("n", [1, 15, 16, 64, 65, 127, 128, 130, 255, 257])
def test_forward_ignores_what_other_requests_hold(n, heads):
    """A request's last tile reads rows of the next request: infinities and NaN there stay there."""
    Hq, Hkv, d = heads
    wl = synth.make_custom([[("i", 3), ("t", 2)], [("t", n)], [("t", 300)]], n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d,
                           hidden=64, seed=100 + n, parts=("B", "V"))
    ref_o, ref_lse = O.attention_forward(wl.layout, wl.q, wl.k, wl.v, Hq, Hkv, wl.softmax_scale)
    ref_abs, _ = O.attention_forward(wl.layout, wl.q, wl.k, _abs_v(wl.v), Hq, Hkv, wl.softmax_scale)
    L, q, k, v = _dev(wl)
    for t, x in ((q, float("nan")), (k, float("inf")), (v, float("nan"))):
        t[:5], t[5 + n:] = x, x
    o, lse, _, _ = avtp.attn_forward(L, q=q, k=k, v=v, softmax_scale=wl.softmax_scale, scores=False)
    torch.cuda.synchronize()
    mine = slice(5, 5 + n)
    _check_o(o.cpu().numpy()[mine], ref_o[mine], ref_abs[mine])
    np.testing.assert_allclose(lse.cpu().numpy()[:, mine], ref_lse[:, mine], rtol=RTOL, atol=ATOL)


@pytest.mark.parametrize("bad", [{"cu_seqlens": [0, 400, 200, 600]}, {"cu_seqlens": [0, -5, 200, 600]},
                                 {"cu_seqlens": [3, 100, 200, 600]}, {"cu_seqlens": [0, 100, 2 ** 30, 600]},
                                 {"img_start": [0, 90, 0]}])
@pytest.mark.parametrize("scores", [False, True])
@pytest.mark.parametrize("repeat", [1, 14])
def test_forward_beside_a_refused_layout(bad, scores, repeat):
    """Up to 32 requests the forward runs beside the layout's validation (repeat 14: more, it
    waits first): offsets validation refuses reach nothing outside the tensors, O, the LSE and
    the scores stay untouched, and the next call is right again."""
    lay = dict(cu_seqlens=[0, 100, 200, 600], img_cu=[0, 1, 2, 3], img_start=[0, 0, 0], img_len=[60, 60, 200])
    if repeat > 1:  # the same three requests again and again
        lay = dict(cu_seqlens=[0] + [600 * i + c for i in range(repeat) for c in (100, 200, 600)],
                   img_cu=list(range(3 * repeat + 1)), img_start=[0] * 3 * repeat, img_len=[60, 60, 200] * repeat)
        bad = {k: v + lay[k][len(v):] for k, v in bad.items()}
    T = lay["cu_seqlens"][-1]
    good = avtp.Layout.from_host(**lay)
    gen = torch.Generator(device="cuda").manual_seed(4)
    q = torch.randn(T, 8, 128, device="cuda", generator=gen).bfloat16()
    k, v = (torch.randn(T, 2, 128, device="cuda", generator=gen).bfloat16() for _ in range(2))
    c = avtp.ForwardCall(good, q=q, k=k, v=v, scores=scores)
    c.run()
    assert avtp.read_device_status(c.workspace) == avtp.OK
    ref = [t.clone() for t in (c.o, c.lse)]
    host = {name: np.asarray({**lay, **bad}[name], dtype=np.int32) for name in lay}
    dev = {name: torch.from_numpy(x.copy()).cuda() for name, x in host.items()}
    b = avtp.ForwardCall(avtp.Layout(host=good.host, **dev), q=q, k=k, v=v, scores=scores, workspace=c.workspace)
    b.o.fill_(7.0), b.lse.fill_(7.0)
    if scores:
        b.scores.fill_(7.0)
    b.run()
    assert avtp.read_device_status(c.workspace) == avtp.ERR_DEVICE_INPUT
    assert torch.all(b.o == 7.0) and torch.all(b.lse == 7.0) and (not scores or torch.all(b.scores == 7.0))
    c.o.zero_(), c.lse.zero_()
    c.run()
    assert avtp.read_device_status(c.workspace) == avtp.OK
    assert torch.equal(c.o, ref[0]) and torch.equal(c.lse, ref[1])
