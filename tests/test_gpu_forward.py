"""Forward-pass numerics of the CUDA kernels against the oracle's network, and the tensor-core
contraction against the FMA kernel and an fp64 product."""
import numpy as np
import pytest
import torch

import tests.parity as parity
from oracle import tsfm_oracle as orc
from tsfm_inputs import Arch, Workload, build_models

pytestmark = pytest.mark.gpu


def small_workload(dtype, target, draft, P=32, mode="separate", patch_in=0):
    return Workload("T", 5, 8 * P, P, 4 * P, 3, 1.0, dtype, target, draft, mode, "c1", series_seed=77,
                    patch_in=patch_in)


def run_forward_case(wl, backend, n_tokens, B=5, seed=0):
    import paper_2511_18191_b200 as tsfm
    tw, dw = build_models(wl)
    dec = tsfm.SpecDecoder(tw, dw, wl.target, wl.draft, wl.patch_len, wl.dtype,
                           "layer_skip" if wl.draft_mode == "layer_skip" else "separate",
                           max_batch=B, max_ctx_tokens=n_tokens, max_horizon_patches=4, max_K=4,
                           gemm_backend=backend, patch_in=wl.patch_in)
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((B, n_tokens, wl.token_len)).astype(np.float32)
    zt = torch.from_numpy(z).cuda()
    got_t = dec.model_forward(0, zt).cpu().numpy()
    got_d = dec.model_forward(1, zt).cpu().numpy()
    dec.close()
    tm, dm = parity.oracle_models(wl, tw, dw)
    want_t = np.stack([orc.forward(tm, z[b].astype(np.float64)) for b in range(B)])
    want_d = np.stack([orc.forward(dm, z[b].astype(np.float64)) for b in range(B)])
    return got_t, want_t, got_d, want_d


@pytest.mark.parametrize("target,draft,P,n", [
    (Arch(2, 128, 4, 512), Arch(1, 64, 2, 256), 96, 7),        # C0's models (head size 32)
    (Arch(2, 128, 2, 256), Arch(1, 128, 1, 128), 32, 21),      # head sizes 64 and 128, several query tiles
    (Arch(1, 128, 2, 256), Arch(1, 64, 2, 128), 32, 197),      # long rows: keys split over a cluster, ragged tail
])
def test_fp32_forward_matches_oracle(target, draft, P, n):
    wl = small_workload("f32", target, draft, P)
    gt, wt, gd, wd = run_forward_case(wl, 0, n)
    assert np.abs(gt - wt).max() < 1e-4
    assert np.abs(gd - wd).max() < 1e-4


@pytest.mark.parametrize("dtype,n", [("f32", 21), ("bf16", 300)])
def test_forced_plain_kernels_are_a_second_implementation(dtype, n):
    """TSFM_GEMM_SIMT shares no contraction kernel with the default path: another order of sums, the same result."""
    import paper_2511_18191_b200 as tsfm
    wl = small_workload(dtype, Arch(1, 128, 2, 256), Arch(1, 128, 1, 128), 32)
    plain, want, _, _ = run_forward_case(wl, tsfm.TSFM_GEMM_SIMT, n)
    auto, _, _, _ = run_forward_case(wl, tsfm.TSFM_GEMM_AUTO, n)
    if dtype == "f32":
        assert np.abs(plain - want).max() < 1e-4
        assert (plain != auto).mean() > 0.1
    else:
        assert parity.value_error("rel_rms", plain, want) < 2e-2
        assert (plain != auto).mean() > 0.1


@pytest.mark.parametrize("target,n", [
    (Arch(1, 64, 1, 64), 2),          # K = 64: two vectors per warp; ten rows of a 16-row tile
    (Arch(1, 64, 2, 128), 150),       # 750 rows: ragged last 16-row tile
    (Arch(1, 320, 5, 768), 60),       # 300 rows x 960 features: 32 x 32 tiles, ragged rows; K = 768 whole and in chunks
    (Arch(1, 832, 13, 832), 3),       # longer rows: chunks of 256 with a short last one
])
def test_fp32_contraction_tiles(target, n):
    wl = small_workload("f32", target, Arch(1, 64, 2, 128), 32)
    gt, wt, gd, wd = run_forward_case(wl, 0, n)
    assert np.abs(gt - wt).max() < 1e-4        # as above: rounding of fp32 sums
    assert np.abs(gd - wd).max() < 1e-4


@pytest.mark.parametrize("target,B", [
    (Arch(1, 64, 1, 128), 182),       # 5460 rows: 258 tiles of 64 x 64 for q, k, v (plain kernel), 172 and 86 for the rest
    (Arch(1, 256, 4, 1024), 138),     # 4140 rows: 1040 tiles of K = 256 for W1 (plain kernel), 780 for q, k, v
    (Arch(1, 512, 8, 512), 23),       # 690 rows: chunks of K; the norm a launch of its own for q, k, v, folded in for W1
    (Arch(1, 512, 8, 512), 16),       # 480 rows: 240 tiles of 32 x 32 with whole rows of 512 for all but q, k, v
])
def test_fp32_contractions_of_many_rows(target, B):
    """Either side of the rule that sends fp32 contractions of many rows to the plain kernel, and of folding norms."""
    wl = small_workload("f32", target, Arch(1, 64, 2, 128), 32)
    gt, wt, gd, wd = run_forward_case(wl, 0, 30, B=B)
    assert np.abs(gt - wt).max() < 1e-4        # as above: rounding of fp32 sums
    assert np.abs(gd - wd).max() < 1e-4


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_forward_of_more_than_two_million_tokens(dtype):
    """8200 windows of 256 tokens: 65600 tiles of 32 rows in the embedding, the head and the fp32 contractions, where
    the y of a grid counts to 65535."""
    import paper_2511_18191_b200 as tsfm
    wl = small_workload(dtype, Arch(1, 64, 1, 64), Arch(1, 64, 1, 64), 16)
    tw, dw = build_models(wl)
    B, n = 8200, 256
    dec = tsfm.SpecDecoder(tw, dw, wl.target, wl.draft, wl.patch_len, wl.dtype, "separate", max_batch=B, max_ctx_tokens=n,
                           max_horizon_patches=1, max_K=1)
    z = torch.randn((B, n, 16), device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    got = dec.model_forward(0, z)
    dec.close()
    tm, _ = parity.oracle_models(wl, tw, dw)
    for b in (0, 4099, 8199):
        want = orc.forward(tm, z[b].cpu().numpy().astype(np.float64))
        if dtype == "f32":
            assert np.abs(got[b].cpu().numpy() - want).max() < 1e-4
        else:
            assert parity.value_error("rel_rms", got[b].cpu().numpy(), want) < 2e-2


@pytest.mark.parametrize("backend", [1, 0], ids=["simt", "tcgen05"])
@pytest.mark.parametrize("target,draft,P,n,mode", [
    (Arch(3, 256, 4, 1024), Arch(2, 128, 4, 256), 96, 9, "separate"),      # few tokens: folded norms, K split
    (Arch(4, 512, 8, 2048), Arch(2, 512, 8, 2048), 32, 37, "layer_skip"),  # 185 tokens, layer-skip draft
    (Arch(4, 512, 8, 2048), Arch(2, 512, 8, 2048), 32, 6, "layer_skip"),   # 30 tokens: one 32-token tile
    (Arch(2, 384, 6, 1536), Arch(1, 128, 2, 256), 96, 3, "separate"),      # 6 heads: 3 feature tiles
    (Arch(2, 256, 4, 1024), Arch(1, 128, 2, 256), 32, 120, "separate"),    # 120 keys: tensor-core attention tiles
    (Arch(2, 256, 4, 1024), Arch(1, 128, 2, 256), 32, 200, "separate"),    # 200 keys: several chunks of the key stream
    (Arch(2, 256, 2, 512), Arch(1, 64, 2, 128), 32, 75, "separate"),       # head sizes 128 and 32, ragged last tile
])
def test_bf16_forward_matches_oracle(backend, target, draft, P, n, mode):
    wl = small_workload("bf16", target, draft, P, mode)
    gt, wt, gd, wd = run_forward_case(wl, backend, n)
    assert parity.value_error("rel_rms", gt, wt) < 2e-2
    assert parity.value_error("rel_rms", gd, wd) < 2e-2


@pytest.mark.parametrize("n", [17, 32, 33, 64, 65, 129])
def test_bf16_attention_tiles_of_queries_and_keys(n):
    """Passes of more than 16 tokens: edges of the 16-query warps, of the two- and four-warp blocks, of the 32-key
    halves and 64-key tiles; head sizes 64 (target) and 32 (draft)."""
    wl = small_workload("bf16", Arch(1, 128, 2, 128), Arch(1, 128, 4, 128), 32)
    gt, wt, gd, wd = run_forward_case(wl, 0, n)
    for got, want in ((gt, wt), (gd, wd)):
        assert np.isfinite(got).all()
        for b in range(got.shape[0]):          # as below: bf16 operands, relative rms 3e-2
            assert np.sqrt(np.mean((got[b] - want[b]) ** 2)) <= 3e-2 * np.sqrt(np.mean(want[b] ** 2))


@pytest.mark.parametrize("target,draft,n", [
    (Arch(3, 256, 2, 512), Arch(2, 128, 4, 128), 103),      # 515 rows: norms folded, rotation of head sizes 128 and 32, 3-row tail
    (Arch(3, 256, 4, 256), Arch(2, 128, 2, 384), 130),      # 650 rows, head size 64; half a feature tile over (N = 384)
    (Arch(2, 128, 2, 128), Arch(2, 192, 3, 192), 620),      # 3100 rows: norms apart; d = 192 takes the other kernels
])
def test_bf16_forward_on_pairs_of_sms(target, draft, n):
    wl = small_workload("bf16", target, draft, 32)
    gt, wt, gd, wd = run_forward_case(wl, 0, n)
    assert np.isfinite(gt).all() and np.isfinite(gd).all()
    assert parity.value_error("rel_rms", gt, wt) < 2e-2       # bf16 operands, as above
    assert parity.value_error("rel_rms", gd, wd) < 2e-2


@pytest.mark.parametrize("dtype,P,P_in,n", [("f32", 16, 1, 70), ("f32", 32, 8, 19), ("bf16", 64, 1, 300), ("bf16", 32, 16, 40)])
def test_forward_with_input_tokens_shorter_than_the_patch(dtype, P, P_in, n):
    """Embedding of P_in-step tokens ([d, P_in] weights; 16-byte loads or element by element) under a
    P-step head: next-patch means at every token."""
    wl = small_workload(dtype, Arch(2, 128, 2, 256), Arch(1, 64, 2, 128), P, patch_in=P_in)
    gt, wt, gd, wd = run_forward_case(wl, 0, n, B=3)
    if dtype == "f32":
        assert np.abs(gt - wt).max() < 1e-4 and np.abs(gd - wd).max() < 1e-4
    else:
        assert parity.value_error("rel_rms", gt, wt) < 2e-2 and parity.value_error("rel_rms", gd, wd) < 2e-2


@pytest.mark.parametrize("M,N,K", [(1, 128, 64), (16, 128, 64), (32, 1536, 512), (160, 512, 2048), (33, 96, 128),
                                   (200, 200, 192), (40, 512, 96), (7, 130, 16), (960, 2048, 512), (300, 384, 1280), (2048, 768, 768)])
def test_tensor_core_gemm_matches_fp64_product_and_fma_kernel(M, N, K):
    import paper_2511_18191_b200 as tsfm
    g = torch.Generator(device="cpu").manual_seed(M * 7 + N)
    A = torch.randn((M, K), generator=g).to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g) / K ** 0.5).to(torch.bfloat16)
    want = (A.double() @ W.double().T).numpy()
    Ad, Wd = A.cuda(), W.cuda()
    outs = {}
    for name, backend in (("simt", tsfm.TSFM_GEMM_SIMT), ("tc", tsfm.TSFM_GEMM_AUTO)):
        Cd = torch.full((M, N), float("nan"), device="cuda")
        tsfm.tsfm_gemm_bf16(torch.cuda.current_stream().cuda_stream, Ad, Wd, Cd, M, N, K, backend)
        torch.cuda.synchronize()
        outs[name] = Cd.cpu().numpy()
        assert np.isfinite(outs[name]).all(), name
        assert np.abs(outs[name] - want).max() < 2e-5 * K ** 0.5 + 1e-5, name
    assert np.abs(outs["tc"] - outs["simt"]).max() < 2e-5 * K ** 0.5 + 1e-5


@pytest.mark.parametrize("M,N,K", [(512, 256, 128), (513, 128, 64), (600, 256, 80), (777, 640, 128), (1500, 384, 1088), (6000, 1024, 256),
                                   (9001, 2304, 64)])
def test_many_token_gemm_matches_fp64_product(M, N, K):
    """The kernel on pairs of SMs (from 513 tokens): half a feature tile over, K that is no whole block or no whole
    ring, ragged token tiles, several tiles per pair."""
    import paper_2511_18191_b200 as tsfm
    g = torch.Generator(device="cpu").manual_seed(M * 13 + N)
    A = torch.randn((M, K), generator=g).to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g) / K ** 0.5).to(torch.bfloat16)
    Cd = torch.full((M, N), float("nan"), device="cuda")
    tsfm.tsfm_gemm_bf16(torch.cuda.current_stream().cuda_stream, A.cuda(), W.cuda(), Cd, M, N, K, tsfm.TSFM_GEMM_AUTO)
    torch.cuda.synchronize()
    got = Cd.cpu().double()
    want = A.double() @ W.double().T
    assert torch.isfinite(got).all()
    assert (got - want).abs().max() < 2e-5 * K ** 0.5 + 1e-5


@pytest.mark.parametrize("M,N,K", [(513, 192, 192), (960, 2112, 512), (2048, 832, 768), (1100, 576, 2048), (5000, 320, 2048),
                                   (9000, 1344, 2048), (4100, 448, 320)])
def test_many_token_gemm_of_odd_widths_matches_fp64_product(M, N, K):
    """Widths that are an odd multiple of 64 (from 513 tokens): every branch of the tile rule of the single-SM kernel."""
    test_many_token_gemm_matches_fp64_product(M, N, K)


@pytest.mark.parametrize("M,N,K", [(1, 128, 64), (16, 130, 64), (32, 1536, 512), (33, 96, 128), (40, 512, 192), (64, 384, 1536),
                                   (128, 1152, 384), (31, 512, 2048), (256, 66, 448), (160, 1536, 512), (319, 512, 512),
                                   (512, 256, 1024), (400, 128, 1536), (512, 144, 2048)])
def test_small_batch_gemm_matches_fp64_product(M, N, K):
    """The kernel that keeps its weight tile in registers (few tokens, K up to 2048): ragged token
    and feature tiles, every k step distribution over its eight warps, and the refusal outside its domain."""
    import paper_2511_18191_b200 as tsfm
    g = torch.Generator(device="cpu").manual_seed(M * 11 + N)
    A = torch.randn((M, K), generator=g).to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g) / K ** 0.5).to(torch.bfloat16)
    Ad, Wd = A.cuda(), W.cuda()
    Cd = torch.full((M, N), float("nan"), device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    if (M, N, K) == (160, 1536, 512):                     # 480 CTAs: more than one wave, not this kernel's job
        with pytest.raises(tsfm.TsfmError) as e:
            tsfm.tsfm_gemm_bf16(s, Ad, Wd, Cd, M, N, K, tsfm.TSFM_GEMM_WS)
        assert e.value.code == tsfm.TSFM_ERR_SHAPE
        return
    tsfm.tsfm_gemm_bf16(s, Ad, Wd, Cd, M, N, K, tsfm.TSFM_GEMM_WS)
    torch.cuda.synchronize()
    got = Cd.cpu().numpy()
    want = (A.double() @ W.double().T).numpy()
    assert np.isfinite(got).all()
    assert np.abs(got - want).max() < 2e-5 * K ** 0.5 + 1e-5


@pytest.mark.parametrize("M,N,K", [(1, 1280, 5120), (3, 130, 4096), (17, 1280, 5120), (64, 3840, 1280), (93, 1024, 4096), (129, 64, 2560),
                                   (500, 192, 80), (512, 5120, 1280), (511, 1280, 5120), (130, 1088, 4352), (510, 320, 2560)])
def test_few_token_gemm_matches_fp64_product(M, N, K):
    """The kernel of up to 512 tokens: K in one piece and split over clusters of every size (8, 8, 8, 2, 6, 8, 1, 1, 3, 4, 4),
    rings that hold K and rings that turn over, half a feature tile, ragged token tiles, K that is no whole block."""
    test_many_token_gemm_matches_fp64_product(M, N, K)


@pytest.mark.parametrize("M,N,K", [(600, 2560, 2048), (600, 256, 2048), (520, 130, 2560), (700, 192, 128), (64, 256, 2048)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_gemm_into_outputs_that_start_on_any_float(M, N, K, offset):
    """Outputs that are not 16-byte aligned: K split in two and in four, rows that are whole float4 and not, K in one piece, and
    the kernel of up to 512 tokens.  The values around the output stay as they are."""
    import paper_2511_18191_b200 as tsfm
    g = torch.Generator(device="cpu").manual_seed(M + N)
    A = torch.randn((M, K), generator=g).to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g) / K ** 0.5).to(torch.bfloat16)
    buf = torch.full((M * N + 8,), float("nan"), device="cuda")
    C = buf[offset:offset + M * N]
    tsfm.tsfm_gemm_bf16(torch.cuda.current_stream().cuda_stream, A.cuda(), W.cuda(), C, M, N, K, tsfm.TSFM_GEMM_AUTO)
    torch.cuda.synchronize()
    assert (C.view(M, N).cpu().double() - A.double() @ W.double().T).abs().max() < 2e-5 * K ** 0.5 + 1e-5
    assert torch.isnan(buf[:offset]).all() and torch.isnan(buf[offset + M * N:]).all()


def test_small_batch_gemm_refuses_outputs_that_it_cannot_store():
    """Pairs of features leave as eight bytes: an output that starts on an odd float is refused on the host, as misaligned
    operands are, and left alone."""
    import paper_2511_18191_b200 as tsfm
    A, W = torch.ones((8, 64), dtype=torch.bfloat16, device="cuda"), torch.ones((16, 64), dtype=torch.bfloat16, device="cuda")
    buf = torch.zeros(132, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    with pytest.raises(tsfm.TsfmError) as e:
        tsfm.tsfm_gemm_bf16(s, A, W, buf[1:129], 8, 16, 64, tsfm.TSFM_GEMM_WS)
    assert e.value.code == tsfm.TSFM_ERR_SHAPE and not buf.any()
    tsfm.tsfm_gemm_bf16(s, A, W, buf[2:130], 8, 16, 64, tsfm.TSFM_GEMM_WS)
    assert (buf[2:130] == 64).all() and not buf[:2].any() and not buf[130:].any()


@pytest.mark.parametrize("n", [2, 4, 26, 102])
def test_bf16_forward_of_wide_models_on_few_tokens(n):
    """Folded norms of up to 512 rows (5 n) in the epilogues of that kernel: the target's QKV, W1 and W2 and the draft's W2 (K =
    1088, 4352 and 2560; half a feature tile over) at every n, the others from 130 rows on, where gemm_ws_kernel has no room
    (the draft's Wo never)."""
    wl = small_workload("bf16", Arch(2, 1088, 17, 4352), Arch(2, 320, 5, 2560), 32)
    gt, wt, gd, wd = run_forward_case(wl, 0, n)
    assert np.isfinite(gt).all() and np.isfinite(gd).all()
    assert parity.value_error("rel_rms", gt, wt) < 2e-2       # bf16 operands, as above
    assert parity.value_error("rel_rms", gd, wd) < 2e-2


@pytest.mark.parametrize("B,n", [(1, 33), (2, 128), (1, 200), (3, 257), (5, 129), (1, 500), (2, 385), (3, 520)])
def test_bf16_attention_of_long_passes(B, n):
    """Heads of 64, more than 32 tokens: blocks of 64 and (the last three) of 128 queries, ragged last blocks and key tiles,
    queries rotated in the kernel (up to 512 rows) or before it.  A NaN in a late token reaches the tokens behind it in its own
    series only, and changes nothing else by a bit."""
    import paper_2511_18191_b200 as tsfm
    wl = small_workload("bf16", Arch(2, 128, 2, 256), Arch(1, 256, 4, 256), 32)
    gt, wt, gd, wd = run_forward_case(wl, 0, n, B=B)
    assert parity.value_error("rel_rms", gt, wt) < 2e-2 and parity.value_error("rel_rms", gd, wd) < 2e-2   # bf16 operands, as above
    tw, dw = build_models(wl)
    dec = tsfm.SpecDecoder(tw, dw, wl.target, wl.draft, wl.patch_len, wl.dtype, "separate", max_batch=B, max_ctx_tokens=n,
                           max_horizon_patches=4, max_K=4)
    z = torch.from_numpy(np.random.default_rng(0).standard_normal((B, n, wl.token_len)).astype(np.float32)).cuda()
    z[B - 1, n - 7] = float("nan")
    got = dec.model_forward(0, z).cpu().numpy()
    dec.close()
    want = gt.copy()
    want[B - 1, n - 7:] = np.nan
    np.testing.assert_array_equal(got, want)


def attention_launches(heads, B, n, tmp_path):
    """(kernel, CTAs, shared memory) of the attention launches of a scoring pass, from the profiler's records."""
    import json
    import paper_2511_18191_b200 as tsfm
    arch = Arch(1, 64 * heads, heads, 64)
    wl = small_workload("bf16", arch, arch, 16, mode="layer_skip")
    dec = tsfm.SpecDecoder(build_models(wl)[0], None, arch, arch, 16, "bf16", "layer_skip", max_batch=B, max_ctx_tokens=n,
                           max_horizon_patches=1, max_K=1)
    z = torch.zeros((B, n, 16), device="cuda")
    dec.model_forward(0, z)
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        dec.model_forward(0, z)
    dec.close()
    prof.export_chrome_trace(str(tmp_path / "t.json"))
    ev = [e for e in json.loads((tmp_path / "t.json").read_text())["traceEvents"] if e.get("cat") == "kernel"]
    if not ev:
        pytest.skip("the profiler records no kernels here")
    return [(e["name"], int(np.prod(e["args"]["grid"])), int(e["args"]["shared memory"])) for e in ev if "attn" in e["name"]]


@pytest.mark.parametrize("heads,B,n", [(4, 1, 520), (4, 12, 380), (4, 13, 380)])
def test_small_attention_grids_do_not_share_sms(heads, B, n, tmp_path):
    """20, 144 and 156 CTAs: up to one per SM each takes more than half of an SM's shared memory."""
    (name, ctas, smem), = attention_launches(heads, B, n, tmp_path)
    assert "attn_mma_kernel" in name and ctas == heads * B * -(-n // 128)
    assert (smem + 1024 > 114 * 1024) == (ctas <= 148)


@pytest.mark.parametrize("B,n,mma", [(16, 33, False), (320, 64, False), (320, 100, False), (320, 160, False), (80, 192, False),
                                     (1, 256, True), (320, 256, True), (320, 380, True)])
def test_blocks_of_128_queries_are_not_given_passes_that_leave_them_empty(B, n, mma, tmp_path):
    """Blocks of 64 queries for windows of up to 100 tokens and up to 1280 pairs, and where a second block of 128 stays half empty;
    blocks of 128 for long passes."""
    (name, _, _), = attention_launches(4, B, n, tmp_path)
    assert ("attn_mma_kernel" in name) == mma and ("attn_tiles_kernel" in name) != mma


@pytest.mark.parametrize("B,n,mma", [(321, 100, True), (640, 80, True), (640, 48, False)])
def test_windows_of_many_series_take_blocks_of_128_queries(B, n, mma, tmp_path):
    """More than 1280 pairs: the waves of blocks decide for short windows too."""
    (name, _, _), = attention_launches(4, B, n, tmp_path)
    assert ("attn_mma_kernel" in name) == mma and ("attn_tiles_kernel" in name) != mma


@pytest.mark.parametrize("n", [103, 205])
def test_bf16_forward_with_k_split_over_two_pairs(n):
    """Residual contractions of 515 and 1025 rows whose K is long and whose tiles are few: two pairs of SMs per tile, each with
    half of K and half of the rows to finish, the last row block ragged or without rows for one of them."""
    wl = small_workload("bf16", Arch(2, 256, 4, 2048), Arch(1, 384, 6, 4096), 32)
    gt, wt, gd, wd = run_forward_case(wl, 0, n)
    assert parity.value_error("rel_rms", gt, wt) < 2e-2       # bf16 operands, as above
    assert parity.value_error("rel_rms", gd, wd) < 2e-2
