"""One decoder layer's attention on its own."""
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
