"""Attention and MLP of one decoder layer on their own, against 64-bit arithmetic that rounds where the bf16 path rounds
(operands, cached keys and values, the attention's output, the MLP's activations).  What is left is the order of fp32 sums, so
that these bounds see what a whole forward pass at 2e-2 cannot: a query that lost its low part, a row factor or a slice of a
folded norm that is off, a partial sum that went astray."""
import math

import numpy as np
import pytest
import torch

from tsfm_inputs import Arch
from tsfm_inputs.weights import make_model, round_to_bf16

pytestmark = pytest.mark.gpu


def layer_weights(arch, rng, **scales):
    """One layer between an embedding and a head that copy their values; scales: standard deviation of a matrix's outputs for
    inputs of size 1 (0: the matrix is zero)."""
    w = make_model(arch, arch.d_model, 0, "bf16")
    w["W_emb"] = w["W_head"] = np.eye(arch.d_model, dtype=np.float32)
    for name in ("Wq", "Wk", "Wv", "Wo", "W1", "W2"):
        t = w["layers.0." + name]
        w["layers.0." + name] = round_to_bf16(rng.standard_normal(t.shape).astype(np.float32) * np.float32(scales[name] / math.sqrt(t.shape[1])))
    for name in ("layers.0.g1", "layers.0.g2", "g_f"):
        w[name] = (1 + 0.2 * rng.standard_normal(arch.d_model)).astype(np.float32)
    return w


def forward(w, arch, z):
    import paper_2511_18191_b200 as tsfm
    B, n, P = z.shape
    dec = tsfm.SpecDecoder(w, None, arch, arch, P, "bf16", "layer_skip", max_batch=B, max_ctx_tokens=n, max_horizon_patches=1,
                           max_K=1)
    got = dec.model_forward(0, torch.from_numpy(z).cuda()).cpu().numpy()
    dec.close()
    return got


def bf16(x):
    return round_to_bf16(np.asarray(x, dtype=np.float32)).astype(np.float64)


def rstd(x):
    return 1 / np.sqrt((x * x).mean(-1, keepdims=True) + 1e-6)


def normed(x, g, folded):
    """What a contraction makes of a normed row: operand and factor."""
    if folded:
        return bf16(g * x.astype(np.float32)), rstd(x)
    return bf16(g * x * rstd(x)), 1.0


def relative(got, want):
    return float(np.sqrt(((got - want) ** 2).mean() / (want ** 2).mean()))


def attention(w, heads, z, round_queries=False):
    """Layer output of x + Wo attention(x) for rows whose norm needs no rounding (all values +1 or -1, gain 1)."""
    x = z.astype(np.float64)
    B, n, d = x.shape
    dh = d // heads
    split = lambda t: t.reshape(B, n, heads, dh).transpose(0, 2, 1, 3)  # noqa: E731
    q, k, v = (split(x * rstd(x) @ w["layers.0." + m].T.astype(np.float64)) for m in ("Wq", "Wk", "Wv"))
    angle = np.arange(n)[:, None] * 1e4 ** (-2.0 * np.arange(dh // 2) / dh)
    c, s = np.cos(angle), np.sin(angle)
    turn = lambda t: np.concatenate([t[..., :dh // 2] * c - t[..., dh // 2:] * s, t[..., dh // 2:] * c + t[..., :dh // 2] * s], -1)  # noqa: E731
    q = turn(q) * (math.log2(math.e) / math.sqrt(dh))
    e = (bf16(q) if round_queries else q) @ bf16(turn(k)).transpose(0, 1, 3, 2)
    e = np.where(np.tril(np.ones((n, n), dtype=bool)), e, -np.inf)
    p = np.exp2(e - e.max(-1, keepdims=True))
    o = p / p.sum(-1, keepdims=True) @ bf16(v)
    y = x + bf16(o.transpose(0, 2, 1, 3).reshape(B, n, d)) @ w["layers.0.Wo"].T.astype(np.float64)
    return y * rstd(y) * w["g_f"]


@pytest.mark.parametrize("B,n", [(1, 20), (2, 33), (3, 64), (2, 100), (1, 129), (2, 200), (2, 300), (3, 384)])
def test_attention_keeps_both_parts_of_its_queries(B, n):
    """Heads of 64 with scores of a few dozen, where a query rounded to bf16 shows.  The bound: probabilities are bf16 (rms error
    of a rounding 2^-9 / sqrt(3) = 1.1e-3, less where several keys share a row)."""
    arch = Arch(1, 128, 2, 64)
    rng = np.random.default_rng(n)
    w = layer_weights(arch, rng, Wq=12, Wk=1, Wv=4, Wo=1, W1=1, W2=0)
    w["layers.0.g1"] = np.ones(128, dtype=np.float32)
    z = np.where(rng.random((B, n, 128)) < 0.5, -1, 1).astype(np.float32)
    want = attention(w, 2, z)
    assert relative(attention(w, 2, z, round_queries=True), want) > 2 * 1.5e-3
    assert relative(forward(w, arch, z), want) < 1.5e-3


@pytest.mark.parametrize("heads,B,n", [(2, 1, 17), (4, 40, 17), (2, 31, 24), (4, 20, 31), (2, 150, 32), (4, 3, 32), (2, 2, 33)])
def test_attention_of_passes_that_see_at_most_32_keys(heads, B, n):
    """Heads of 64 and 32 at the ends of 17 to 32 tokens, few and many series (rotated here or by the contraction).  The bound as
    above."""
    arch = Arch(1, 128, heads, 64)
    rng = np.random.default_rng(n + heads)
    w = layer_weights(arch, rng, Wq=12, Wk=1, Wv=4, Wo=1, W1=1, W2=0)
    w["layers.0.g1"] = np.ones(128, dtype=np.float32)
    z = np.where(rng.random((B, n, 128)) < 0.5, -1, 1).astype(np.float32)
    assert relative(forward(w, arch, z), attention(w, heads, z)) < 1.5e-3


@pytest.mark.parametrize("d,f,B,n,folded", [
    (192, 192, 1, 3, True),           # weights in registers
    (256, 2560, 4, 20, True),         # up to 512 rows: K of W2 split over a cluster
    (128, 4352, 5, 101, True),        # 505 rows
    (256, 1024, 5, 103, True),        # pairs of SMs, several row blocks, the last one ragged
    (256, 4096, 5, 103, True),        # K of W2 split over two pairs
    (128, 2048, 5, 205, True),        # the same, half a feature tile over
    (192, 320, 4, 150, False),        # odd multiples of 64: the kernel on one SM, norm apart
    (256, 512, 8, 500, False),        # 4000 rows: norms apart, several tiles per pair
])
def test_mlp_of_a_layer(d, f, B, n, folded):
    """x + W2 GELU(W1 norm(x)).  The bound: fp32 sums of relative error 1e-6 round to the other bf16 neighbour, 2^-8 away, in 5 of
    ten thousand activations (rms 9e-5 of what the MLP adds)."""
    arch = Arch(1, d, d // 64, f)
    rng = np.random.default_rng(f + n)
    w = layer_weights(arch, rng, Wq=1, Wk=1, Wv=1, Wo=0, W1=1.5, W2=4)
    z = (rng.standard_normal((B, n, d)) * np.exp(rng.standard_normal((B, n, 1)))).astype(np.float32)
    x = z.astype(np.float64)
    a, k = normed(x, w["layers.0.g2"], folded)
    h = torch.from_numpy(a @ w["layers.0.W1"].T.astype(np.float64) * k)
    y = x + bf16(torch.nn.functional.gelu(h).numpy()) @ w["layers.0.W2"].T.astype(np.float64)
    assert relative(forward(w, arch, z), y * rstd(y) * w["g_f"]) < 1.5e-4


@pytest.mark.parametrize("half", [0, 1])
@pytest.mark.parametrize("f,B,n", [(512, 9, 500), (2048, 19, 331)])
def test_mlp_of_a_layer_with_folded_norms_and_several_tiles_per_pair(f, B, n, half):
    """4500 and 6289 rows of 512 values (the token and the token halved; the head reads one of the two): the last row block in
    part, accumulators used in turn.  The bound as above."""
    d, P = 512, 256
    arch = Arch(1, d, d // 64, f)
    rng = np.random.default_rng(f + n)
    w = layer_weights(arch, rng, Wq=1, Wk=1, Wv=1, Wo=0, W1=1.5, W2=4)
    eye = np.eye(P, dtype=np.float32)
    w["W_emb"], w["W_head"] = np.concatenate([eye, eye / 2]), np.concatenate([eye * (half == 0), eye * (half == 1)], 1)
    z = (rng.standard_normal((B, n, P)) * np.exp(rng.standard_normal((B, n, 1)))).astype(np.float32)
    x = np.concatenate([z, z / 2], -1).astype(np.float64)
    a, k = normed(x, w["layers.0.g2"], True)
    h = torch.from_numpy(a @ w["layers.0.W1"].T.astype(np.float64) * k)
    y = x + bf16(torch.nn.functional.gelu(h).numpy()) @ w["layers.0.W2"].T.astype(np.float64)
    want = y * rstd(y) * w["g_f"]
    assert relative(forward(w, arch, z), want[..., half * P:half * P + P]) < 1.5e-4


def embedding_and_head_error(d, P, P_in, B, n):
    arch = Arch(1, d, d // 64, 64)
    rng = np.random.default_rng(d + n)
    w = make_model(arch, P, 1, "bf16", patch_in=P_in)
    for name in ("Wo", "W2"):
        w["layers.0." + name][:] = 0
    w["g_f"] = (1 + 0.2 * rng.standard_normal(d)).astype(np.float32)
    import paper_2511_18191_b200 as tsfm
    z = rng.standard_normal((B, n, P_in)).astype(np.float32)
    dec = tsfm.SpecDecoder(w, None, arch, arch, P, "bf16", "layer_skip", max_batch=B, max_ctx_tokens=max(n, 2 * P // P_in),
                           max_horizon_patches=1, max_K=1, patch_in=P_in)
    got = dec.model_forward(0, torch.from_numpy(z).cuda()).cpu().numpy()
    dec.close()
    x = z.astype(np.float64) @ w["W_emb"].T.astype(np.float64)
    return relative(got, (w["g_f"] * x * rstd(x)) @ w["W_head"].T.astype(np.float64))


@pytest.mark.parametrize("d,P,P_in,B,n", [
    (64, 16, 16, 9, 60),              # 540 rows: operands in registers
    (192, 48, 48, 5, 103),            # half a block of k, a ragged tile of rows
    (128, 80, 80, 3, 43),             # 129 rows: embedding row by row, head tiled (in registers)
    (1280, 32, 32, 64, 9),            # five chunks of a row
    (320, 256, 16, 2, 320),           # a chunk and a quarter; 192 + 64 features
    (832, 96, 96, 200, 27),           # 5400 rows: 96 and 192 features a CTA
])
def test_embedding_and_head_are_exact_to_fp32(d, P, P_in, B, n):
    """Layers that add nothing between embedding, final norm and head of a bf16 model, whose rows are fp32.  The bound: sums of
    up to 1280 products in blocks of 32, fp32 rounding (relative 2^-24 each) in embedding, square, factor and head: measured
    1.0e-7 to 1.3e-7, and an operand that lost its last 8 bits shows as 2^-17 = 8e-6."""
    assert embedding_and_head_error(d, P, P_in, B, n) < 3e-7


@pytest.mark.parametrize("d,P,P_in,B,n", [
    (64, 256, 256, 9, 60), (192, 16, 16, 9, 60),   # 540 rows: tiles of 16 and 8 features
    (192, 80, 80, 3, 43),                          # embedding row by row
    (64, 16, 16, 60, 200),                         # rows of half a block of k
    (64, 48, 48, 17, 104), (64, 48, 48, 17, 105),  # embeddings of 444 and 448 tiles of 16 x 16
    (64, 96, 96, 25, 47), (64, 96, 96, 25, 48),    # heads of 444 and 450
    (128, 112, 112, 37, 16), (128, 112, 112, 37, 17),   # embeddings of 296 and 320
])
def test_tiles_of_embedding_and_head(d, P, P_in, B, n):
    """Both sides of the line between operands in registers and rows in three parts.  The bound as above."""
    assert embedding_and_head_error(d, P, P_in, B, n) < 1.3 * math.hypot(math.sqrt(P_in / 2) * 2.5e-8, 1.1e-7)


@pytest.mark.parametrize("d,P,P_in,B,n", [
    (128, 96, 96, 1, 31), (128, 96, 96, 2, 16),                  # row by row and four rows a block
    (192, 32, 32, 3, 11), (64, 176, 176, 5, 7), (320, 160, 160, 67, 7),   # ragged rows and features
    (128, 16, 1, 3, 37), (128, 16, 4, 25, 43),                   # tokens shorter than a vector, folded and not
])
def test_embedding_of_few_rows(d, P, P_in, B, n):
    """The bound as above: here the embedding is one chain of up to 176 sums, whose roundings (0.42 x 2^-24 of a partial sum in the
    mean square) add up to sqrt(176 / 2) x 2.5e-8 = 2.4e-7, with the rest 2.6e-7."""
    test_embedding_and_head_are_exact_to_fp32(d, P, P_in, B, n)


@pytest.mark.parametrize("d,P,P_in,B,n", [
    (512, 176, 176, 3, 11), (320, 256, 256, 4, 40),              # more shared memory than a kernel has by itself
    (640, 64, 8, 3, 23), (192, 48, 16, 35, 17), (64, 64, 8, 7, 81),   # one and two vectors in registers, folded and not
])
def test_embedding_of_four_rows(d, P, P_in, B, n):
    """The chain's sqrt(P_in / 2) x 2.5e-8 (as above, 2.8e-7 for 256 values) and 1.1e-7 for the rest are the error to expect, its root
    mean square over some thousand values; the bound is 1.3 times that."""
    assert embedding_and_head_error(d, P, P_in, B, n) < 1.3 * math.hypot(math.sqrt(P_in / 2) * 2.5e-8, 1.1e-7)


@pytest.mark.parametrize("d,f,P,P_in,B,n", [
    (64, 64, 64, 64, 1, 1), (64, 64, 48, 48, 1, 17), (64, 64, 16, 16, 10, 16), (64, 64, 16, 16, 7, 23),   # up to 160 rows
    (64, 64, 32, 8, 5, 3),                                       # embedding by itself
    (128, 128, 128, 128, 1, 15), (128, 64, 112, 112, 4, 16), (128, 128, 80, 16, 5, 13), (64, 128, 96, 96, 2, 9),   # up to 64
    (192, 128, 64, 64, 1, 33),                                   # a wider model: W2 only
])
def test_fp32_links_of_few_rows(d, f, P, P_in, B, n):
    """x + W2 GELU(W1 norm(x)), norm and head of an fp32 model.  The bound: five links of up to 192 products in tree sums,
    each with up to ten roundings of relative size 2^-24 that add as the square root: 4e-7."""
    arch = Arch(1, d, d // 32, f)
    rng = np.random.default_rng(d + n)
    w = make_model(arch, P, 1, "f32", patch_in=P_in)
    w["layers.0.Wo"][:] = 0
    w["layers.0.W1"] *= 3
    for name in ("g_f", "layers.0.g2"):
        w[name] = (1 + 0.2 * rng.standard_normal(d)).astype(np.float32)
    import paper_2511_18191_b200 as tsfm
    z = rng.standard_normal((B, n, P_in)).astype(np.float32)
    dec = tsfm.SpecDecoder(w, None, arch, arch, P, "f32", "layer_skip", max_batch=B, max_ctx_tokens=max(n, 2 * P // P_in),
                           max_horizon_patches=1, max_K=1, patch_in=P_in)
    got = dec.model_forward(0, torch.from_numpy(z).cuda()).cpu().numpy()
    dec.close()
    x = z.astype(np.float64) @ w["W_emb"].T.astype(np.float64)
    h = torch.from_numpy((w["layers.0.g2"] * x * rstd(x)) @ w["layers.0.W1"].T.astype(np.float64))
    y = x + torch.nn.functional.gelu(h).numpy() @ w["layers.0.W2"].T.astype(np.float64)
    assert relative(got, (w["g_f"] * y * rstd(y)) @ w["W_head"].T.astype(np.float64)) < 4e-7


@pytest.mark.parametrize("heads,B,n", [(4, 9, 60), (1, 9, 60), (4, 2, 300), (1, 2, 300), (2, 9, 142), (2, 9, 143), (2, 41, 251)])
def test_rotation_in_the_contraction_of_passes_of_many_tokens(heads, B, n):
    """Heads of 32, 64 and 128, the rotation table of a pass in shared memory or not, ragged row blocks, several tiles per pair.
    The bound as above."""
    arch = Arch(1, 128, heads, 64)
    rng = np.random.default_rng(n + heads)
    w = layer_weights(arch, rng, Wq=8, Wk=1, Wv=4, Wo=1, W1=1, W2=0)
    w["layers.0.g1"] = np.ones(128, dtype=np.float32)
    z = np.where(rng.random((B, n, 128)) < 0.5, -1, 1).astype(np.float32)
    assert relative(forward(w, arch, z), attention(w, heads, z)) < 1.5e-3


@pytest.mark.parametrize("heads,n,late", [
    (2, 20, 3), (4, 32, 9), (1, 31, 1),          # blocks of two warps, head sizes 64, 32 and 128
    (2, 40, 7), (4, 100, 40), (1, 70, 2),        # blocks of four
    (2, 200, 150), (2, 200, 5),                  # a value in a tile that all later queries see, and in one that some see
    (2, 400, 7), (2, 400, 390), (2, 400, 140),   # blocks of 128 queries
])
@pytest.mark.parametrize("kind", ["infinite", "nan"])
def test_values_reach_only_the_queries_that_see_them(heads, n, late, kind):
    """One token whose value vector holds an infinity (its key is finite) or that is NaN altogether: NaN from that token on in
    its series, not a bit of difference before it and in the other series."""
    arch = Arch(1, 128, heads, 64)
    rng = np.random.default_rng(n)
    w = layer_weights(arch, rng, Wq=8, Wk=1, Wv=1, Wo=1, W1=1, W2=0)
    w["layers.0.g1"] = np.ones(128, dtype=np.float32)
    z = np.where(rng.random((2, n, 128)) < 0.5, -1, 1).astype(np.float32)
    j = n - late
    z[0, j] = np.eye(128)[5] if kind == "infinite" else np.nan      # normed, its sixth feature is sqrt(128)
    w["layers.0.Wo"][:, 0] = 0
    w["layers.0.Wv"][0] = 0
    want = forward(w, arch, np.nan_to_num(z))
    assert np.isfinite(want).all()
    if kind == "infinite":
        w["layers.0.Wv"][0, 5] = round_to_bf16(np.array([3.1e37]))[0]   # 3.5e38 for that token, 3.1e37 for the others
    want[0, j:] = np.nan
    np.testing.assert_array_equal(forward(w, arch, z), want)
