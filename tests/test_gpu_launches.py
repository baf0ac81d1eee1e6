"""Which kernel a call launches and how large, from the profiler's records: choices that change no result.  (In a file behind those whose
oracle runs fork worker processes: a profiler session before a fork leaves later ones without records.)"""
import json

import numpy as np
import pytest
import torch

from tests.gpu_common import make_decoder, series_on_device
from tsfm_inputs import Arch, workload
from tsfm_inputs.weights import make_model

pytestmark = pytest.mark.gpu


def launches(call, part, tmp_path):
    """(name, grid, block) of the kernels of a second call whose names hold `part`."""
    call()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
    prof.export_chrome_trace(str(tmp_path / "t.json"))
    ev = [e for e in json.loads((tmp_path / "t.json").read_text())["traceEvents"] if e.get("cat") == "kernel"]
    if not ev:
        pytest.skip("the profiler records no kernels here")
    return [(e["name"], e["args"]["grid"], e["args"]["block"]) for e in ev if part in e["name"]]


@pytest.mark.parametrize("heads,ctx,K", [(4, 8, 17), (2, 8, 17), (2, 5, 17)])
def test_bounds_checking_mode_takes_the_same_attention_kernels(heads, ctx, K, tmp_path):
    """Verification passes whose capacity is 32 tokens or less, one more with the spare token of that mode."""
    import paper_2511_18191_b200 as tsfm
    wl = workload("C1", batch=9, ctx_len=32 * ctx, patch_len=32, horizon=32 * 6, K=K, target=Arch(2, 128, heads, 256), draft=Arch(1, 128, heads, 256))
    _, series = series_on_device(wl)
    names = []
    for mode in (0, tsfm.TSFM_EXEC_CHECK_BOUNDS):
        dec = make_decoder(wl, max_K=K, exec_mode=tsfm.TSFM_EXEC_STREAM | mode)[0]
        names.append({name for name, _, _ in launches(lambda: dec.forecast(series, wl.horizon, K, 3.0, 17), "attn", tmp_path)})
        dec.close()
    assert names[0] == names[1] and any("attn_short_kernel" in name for name in names[0])


@pytest.mark.parametrize("B,K", [(300, 7), (1100, 1), (3000, 7), (5000, 3)])
def test_acceptance_step_is_resident_at_once(B, K, tmp_path):
    """32 warps on an SM, or one per series; whole CTAs of eight."""
    import paper_2511_18191_b200 as tsfm
    wl = workload("C0", batch=B, series_recipe="c1", ctx_len=64, patch_len=16, horizon=16 * 3, K=K, target=Arch(1, 64, 1, 64), draft=Arch(1, 64, 2, 64))
    _, series = series_on_device(wl)
    dec = make_decoder(wl, max_K=K, exec_mode=tsfm.TSFM_EXEC_STREAM)[0]
    got = launches(lambda: dec.forecast(series, wl.horizon, K, 1.5, 5), "accept_kernel", tmp_path)
    dec.close()
    assert got and all(np.prod(grid) * np.prod(block) < 32 * (max(32 * 148, B) + 8) for _, grid, block in got)


@pytest.mark.parametrize("dtype,simt,d,P,P_in,B,n,rows", [
    ("f32", 1, 64, 96, 96, 11, 100, 4), ("f32", 1, 128, 256, 256, 11, 100, 4), ("bf16", 1, 256, 176, 176, 11, 100, 4),   # many rows
    ("bf16", 0, 256, 256, 256, 4, 25, 4), ("bf16", 0, 512, 32, 32, 4, 8, 4), ("bf16", 0, 512, 32, 32, 1, 31, 1),
    ("bf16", 0, 64, 96, 96, 4, 25, 1), ("bf16", 0, 128, 16, 16, 4, 80, 1),       # few rows of narrow models
])
def test_rows_that_share_an_embedding_cta(dtype, simt, d, P, P_in, B, n, rows, tmp_path):
    import paper_2511_18191_b200 as tsfm
    arch = Arch(1, d, d // 32, 64)
    dec = tsfm.SpecDecoder(make_model(arch, P, 1, dtype, patch_in=P_in), None, arch, arch, P, dtype, "layer_skip", max_batch=B, max_ctx_tokens=n,
                           max_horizon_patches=1, max_K=1, patch_in=P_in, gemm_backend=tsfm.TSFM_GEMM_SIMT if simt else tsfm.TSFM_GEMM_AUTO)
    z = torch.zeros((B, n, P_in), device="cuda")
    (_, grid, _), = launches(lambda: dec.model_forward(0, z), "embed_kernel", tmp_path)
    dec.close()
    assert grid == [-(-B * n // rows), -(-d // 128), 1]
