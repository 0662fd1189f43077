"""The text-attention criterion's tensor-core passes at their edges, against the fp64 oracle:
key tiles of 128 and their remainders, row blocks of 256 and their halves, runs of a CTA that
cross blocks, first visible rows inside a 32-row chunk, and a softmax reference that moves.
"""
import ctypes

import numpy as np
import pytest
import torch

from oracle import avtp_oracle as O
from paper_2608_26806_gb300 import avtp, synth
from tests.gpu_util import assert_scores_close, bf16_dev, dev_layout, ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ensure_built()


def _check(wl, scale=None, lse=None):
    Hq, Hkv = wl.n_q_heads, wl.n_kv_heads
    scale = wl.softmax_scale if scale is None else scale
    L = dev_layout(wl.layout)
    scores, sums = avtp.score(L, "text_attention", q=bf16_dev(wl.q), k=bf16_dev(wl.k), softmax_scale=scale, lse=lse,
                              path="tensor")
    torch.cuda.synchronize()
    got = scores.cpu().numpy()
    ref = O.score_text_attention(wl.layout, wl.q, wl.k, Hq, Hkv, scale)
    assert_scores_close(got, ref, wl.layout.visual_mask())
    assert np.array_equal(sums.cpu().numpy(), O.image_sums(wl.layout, got))


_LAYOUTS = {
    # image sizes about a key tile, one text token between the images (G rows each)
    "tiles": [[("t", 2)] + [s for n in (1, 127, 128, 129, 255, 256, 257, 2) for s in (("i", n), ("t", 1))]],
    # more row blocks than CTAs have steps: runs that cross several blocks
    "blocks": [[("i", 130), ("t", 500)], [("t", 40), ("i", 3), ("t", 300)], [("i", 64), ("t", 129)]] * 3,
    # requests whose rows end in the first half, at the half, and just past the block
    "halves": [[("i", 200), ("t", n)] for n in (1, 31, 32, 33, 63, 64, 65, 128)],
}


@pytest.mark.parametrize("layout", sorted(_LAYOUTS))
@pytest.mark.parametrize("heads", [(4, 1, 64), (8, 2, 128), (14, 2, 128)])
def test_text_passes_edges(layout, heads):
    Hq, Hkv, d = heads
    _check(synth.make_custom(_LAYOUTS[layout], n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, hidden=64, seed=11,
                             parts=("B",)))


@pytest.mark.parametrize("growth", [40.0, -40.0])
@pytest.mark.parametrize("heads", [(4, 2, 64), (8, 2, 128)])
def test_text_passes_moving_reference(heads, growth):
    """Logits that climb or fall by 40 over 500 keys move a row's reference again and again."""
    Hq, Hkv, d = heads
    wl = synth.make_custom([[("t", 3), ("i", 700), ("t", 90)], [("i", 260), ("t", 129)]], n_q_heads=Hq, n_kv_heads=Hkv,
                           head_dim=d, hidden=64, seed=78, parts=("B",))
    T = wl.layout.n_tokens
    rng = np.random.default_rng(6)
    ramp = growth * (np.arange(T) // 37) * 37 / 500.0
    q = (np.full((T, Hq, d), 1.0 / d) + 0.002 * rng.standard_normal((T, Hq, d))).astype(np.float32)
    k = (ramp[:, None, None] + rng.standard_normal((T, Hkv, d))).astype(np.float32)
    wl.tensors["q"] = synth.f32_to_bf16_bits(q.reshape(T, -1)).reshape(T, Hq, d)
    wl.tensors["k"] = synth.f32_to_bf16_bits(k.reshape(T, -1)).reshape(T, Hkv, d)
    _check(wl, scale=1.0)


# ---------------------------------------------------------------- rows that a key is not scored by
@pytest.mark.parametrize("heads", [(4, 2, 64), (8, 2, 128), (14, 2, 128)])
@pytest.mark.parametrize("fill", [-np.inf, np.nan, np.inf])
def test_normaliser_of_rows_before_an_image(heads, fill):
    """A supplied normaliser counts for the images its query follows alone: one filled in behind
    the first image only scores every image, and a query without one spoils the image before it
    and not the image behind it."""
    Hq, Hkv, d = heads
    wl = synth.make_custom([[("t", 5), ("i", 40), ("t", 37), ("i", 130), ("t", 3), ("i", 9), ("t", 60)],
                            [("t", 70), ("i", 140), ("t", 9)]], n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, hidden=64,
                           seed=21, parts=("B",))
    lay = wl.layout
    lse = O.text_lse(lay, wl.q, wl.k, Hq, Hkv, wl.softmax_scale).astype(np.float32)
    ref = O.score_text_attention(lay, wl.q, wl.k, Hq, Hkv, wl.softmax_scale, lse=lse.astype(np.float64))
    second = int(lay.cu_seqlens[1])
    lse[:, :5] = fill
    lse[:, second:second + 70] = fill
    L, q, k = dev_layout(lay), bf16_dev(wl.q), bf16_dev(wl.k)

    def run(x):
        scores, _ = avtp.score(L, "text_attention", q=q, k=k, softmax_scale=wl.softmax_scale, path="tensor",
                               lse=torch.from_numpy(x).cuda())
        return scores.cpu().numpy()

    assert_scores_close(run(lse), ref, lay.visual_mask())
    lse[:, 45 + 36] = np.nan  # the last query between the first two images
    got, vis = run(lse), lay.visual_mask()
    assert np.all(np.isnan(got[5:45]))
    vis[5:45] = False
    assert_scores_close(got, ref, vis)


@pytest.mark.parametrize("heads", [(4, 2, 64), (3, 1, 128), (8, 2, 128)])
@pytest.mark.parametrize("n", [1, 15, 16, 31, 32, 33, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("how", ["own", "lse", "forward"])
def test_scores_ignore_what_other_requests_hold(heads, n, how):
    """A request's last row block reads rows of the next request: infinities and NaN there stay there."""
    Hq, Hkv, d = heads
    wl = synth.make_custom([[("i", 3), ("t", 2)], [("i", 70), ("t", 1), ("i", 30), ("t", n)], [("i", 40), ("t", 300)]],
                           n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, hidden=64, seed=100 + n, parts=("B", "V"))
    lay, scale = wl.layout, wl.softmax_scale
    a, b = int(lay.cu_seqlens[1]), int(lay.cu_seqlens[2])
    lse = O.text_lse(lay, wl.q, wl.k, Hq, Hkv, scale).astype(np.float32)
    ref = O.score_text_attention(lay, wl.q, wl.k, Hq, Hkv, scale)
    L, q, k = dev_layout(lay), bf16_dev(wl.q), bf16_dev(wl.k)
    lse = torch.from_numpy(lse).cuda()
    for t, x in ((q, float("nan")), (k, float("inf"))):
        t[:a], t[b:] = x, x
    lse[:, :a], lse[:, b:] = float("nan"), float("nan")
    if how == "forward":
        _, _, scores, sums = avtp.attn_forward(L, q=q, k=k, v=bf16_dev(wl.v), softmax_scale=scale, path="tensor")
    else:
        scores, sums = avtp.score(L, "text_attention", q=q, k=k, softmax_scale=scale, path="tensor",
                                  lse=lse if how == "lse" else None)
    got = scores.cpu().numpy()
    mine = lay.visual_mask() & (np.arange(lay.n_tokens) >= a) & (np.arange(lay.n_tokens) < b)
    assert_scores_close(got, ref, mine)
    assert np.array_equal(sums.cpu().numpy()[1:3], O.image_sums(lay, got)[1:3])


@pytest.mark.parametrize("supplied", [False, True])
def test_scores_with_a_loose_text_bound(supplied):
    """Rows between the batch's text and a looser bound on it are workspace nothing has written."""
    Hq, Hkv, d = 8, 2, 128
    wl = synth.make_custom([[("i", 140), ("t", 30)], [("t", 2), ("i", 70), ("t", 41)]], n_q_heads=Hq, n_kv_heads=Hkv,
                           head_dim=d, hidden=64, seed=8, parts=("B",))
    lay, scale = wl.layout, wl.softmax_scale
    lse = O.text_lse(lay, wl.q, wl.k, Hq, Hkv, scale).astype(np.float32)
    ref = O.score_text_attention(lay, wl.q, wl.k, Hq, Hkv, scale)
    L, q, k, lse = dev_layout(lay), bf16_dev(wl.q), bf16_dev(wl.k), torch.from_numpy(lse).cuda()
    for bound in (0, 100, lay.n_tokens):
        sa = avtp._score_args("text_attention", q=q, k=k, softmax_scale=scale, lse=lse if supplied else None,
                              max_text_tokens=bound, path="tensor")
        cl, size = L.c(), ctypes.c_size_t()
        lib = avtp.load()
        assert lib.avtp_workspace_size(ctypes.byref(cl), ctypes.byref(sa), ctypes.byref(size)) == avtp.OK
        ws = torch.full((size.value,), 0xFF, dtype=torch.uint8, device="cuda")
        scores = torch.zeros(lay.n_tokens, device="cuda")
        sums = torch.zeros(lay.n_images, dtype=torch.int64, device="cuda")
        assert lib.avtp_score(ctypes.byref(cl), ctypes.byref(sa), scores.data_ptr(), sums.data_ptr(), ws.data_ptr(),
                              size.value, avtp._stream(None)) == avtp.OK
        torch.cuda.synchronize()
        assert avtp.read_device_status(ws) == avtp.OK
        assert_scores_close(scores.cpu().numpy(), ref, lay.visual_mask())


def test_mass_of_one_key_over_very_many_queries():
    """Every row of a request puts all of its mass on one key: 2^23 rows, whose sum at 40 fraction
    bits would reach the accumulator's top bit. The score is 1."""
    Hq, d, n_text = 128, 64, 65536
    L = avtp.Layout.from_host([0, 1 + n_text], [0, 1], [0], [1])
    q = torch.zeros(1 + n_text, Hq, d, device="cuda", dtype=torch.bfloat16)
    q[:, :, 0] = 1.0
    k = torch.zeros(1 + n_text, 1, d, device="cuda", dtype=torch.bfloat16)
    k[0, 0, 0] = 4.0
    lse = torch.full((Hq, 1 + n_text), 4.0, device="cuda")  # the logit of the image's only token: probability 1
    scores, sums = avtp.score(L, "text_attention", q=q, k=k, softmax_scale=1.0, lse=lse, path="tensor")
    # lse2 and z2 are products of 4 with log2(e), each rounded once: within 2^-20 of each other
    assert abs(float(scores[0]) - 1.0) < 4e-6
    assert abs(int(sums[0]) - 2 ** 32) < 4e-6 * 2 ** 32


@pytest.mark.parametrize("bad", [{"cu_seqlens": [0, 900, 200]}, {"cu_seqlens": [0, -5, 200]},
                                 {"cu_seqlens": [7, 100, 200]}, {"img_start": [0, 180]}, {"img_len": [60, 0]}])
def test_last_token_logits_beside_a_refused_layout(bad):
    """The last-token logits run beside the layout's validation: offsets it refuses (decreasing,
    negative, past the batch, spans outside their request) reach no memory outside the tensors
    and leave the scores and sums untouched."""
    lay = dict(cu_seqlens=[0, 100, 200], img_cu=[0, 1, 2], img_start=[0, 0], img_len=[60, 60])
    good = avtp.Layout.from_host(**lay)
    q = torch.randn(200, 8, 128, device="cuda").bfloat16()
    k = torch.randn(200, 2, 128, device="cuda").bfloat16()
    args = dict(q=q, k=k, query_set="last")
    ws = avtp.new_workspace(avtp.workspace_size(good, "text_attention", **args) + 65536)
    ref, _ = avtp.score(good, "text_attention", workspace=ws, **args)
    host = {name: np.asarray({**lay, **bad}[name], dtype=np.int32) for name in lay}
    dev = {name: torch.from_numpy(v.copy()).cuda() for name, v in host.items()}
    # the host copies keep the good counts, as a caller's would
    L = avtp.Layout(host=good.host, **dev)
    scores = torch.full((200,), 7.0, device="cuda")
    avtp.score(L, "text_attention", workspace=ws, scores=scores, **args)
    assert avtp.read_device_status(ws) == avtp.ERR_DEVICE_INPUT
    assert torch.all(scores == 7.0)
    again, _ = avtp.score(good, "text_attention", workspace=ws, **args)
    assert avtp.read_device_status(ws) == avtp.OK and torch.equal(ref, again)
