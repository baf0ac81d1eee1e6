"""The decoder's work as its users have it: forecasts and scoring passes over the repository's own model shapes.

A case is one call.  `family` names the models (the workload shapes of tsfm_inputs), `op` the entry point:

  spec     speculative forecast (draft K patches, verify them in one pass, accept / correct), the product's main call
  target   plain patch-autoregressive forecast with the target
  forward  one causal pass of the target over whole windows, next-patch means at every token (scoring)

`host` cases start from and end in host memory (the *_host entry points), `stats` cases ask for the call's statistics
and therefore wait for it; the others only enqueue, as a serving loop does.

Weights are random.  `target` and `forward` cases and the fp32 models use Xavier-normal weights.  Speculative decoding
is used with a draft that tracks its target, so the bf16 speculative cases build such pairs: a layer-skip draft whose
missing layers contribute little, a perturbed copy, or two separate models that share a persistence forecast (embedding
and head of both reproduce the last patch, the layers add a correction that the models do not share).  The
temperatures make such a draft pass at the rates that the method is reported with, about nine in ten.
"""
import math

import torch

import paper_2511_18191_b200 as tsfm

# layers, d_model, heads, d_ff of target and draft; P steps per patch, P_in per input token; how the draft relates to
# the target; the temperature; the largest batch, context, horizon (in patches) and block size in use
FAMILIES = {
    # the smallest models, fp32, one series at a time or a few dozen (prototyping, reference runs)
    "c0": dict(target=(2, 128, 4, 512), draft=(1, 64, 2, 256), dtype="f32", P=96, P_in=0, mode="separate", tau=2.0,
               B=64, ctx=30, T=15, K=4),
    # a 25 M-parameter model with a layer-skip draft: from one interactive series to a batch of channels
    "c1": dict(target=(8, 512, 8, 2048), draft=(2, 512, 8, 2048), dtype="bf16", P=96, P_in=0, mode="layer_skip",
               tau=0.2, B=32, ctx=30, T=15, K=8),
    # a 300 M-parameter model with a small separate draft, channels of wide multivariate sets batched
    "c2": dict(target=(24, 1024, 16, 4096), draft=(2, 256, 4, 1024), dtype="bf16", P=96, P_in=0, mode="separate",
               tau=0.3, B=256, ctx=30, T=8, K=8),
    # very many short series
    "c3": dict(target=(12, 768, 12, 3072), draft=(12, 768, 12, 3072), dtype="bf16", P=96, P_in=0, mode="perturbed",
               tau=0.3, B=1024, ctx=7, T=15, K=8),
    # a 500 M-parameter model, long context, long horizon
    "c4": dict(target=(24, 1280, 20, 5120), draft=(4, 384, 6, 1536), dtype="bf16", P=32, P_in=0, mode="separate",
               tau=0.3, B=64, ctx=256, T=64, K=8),
    # point tokens under a 64-step head: many tokens per series and per verification pass
    "c5": dict(target=(6, 512, 8, 2048), draft=(2, 256, 4, 1024), dtype="bf16", P=64, P_in=1, mode="separate",
               tau=0.3, B=16, ctx=12, T=6, K=3),
}
LATE_LAYERS = 0.03        # factor on Wo, W2 of the target layers that a layer-skip draft lacks
PERTURBATION = 0.03       # of a perturbed draft, in standard deviations of each matrix
CORRECTION = 0.1          # factor on Wo, W2 of two separate models around a shared persistence forecast
POINT_CORRECTION = 0.25   # (with point tokens)
POINT_HEAD = 0.1          # and, with point tokens, the share of an ordinary random head in theirs


def _case(name, family, op, B, ctx, H=0, K=0, host=False, stats=False):
    """ctx in patches, H in steps."""
    c = dict(family=family, op=op, B=B, ctx=ctx, H=H, K=K, host=host, stats=stats)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one series, smallest models: the shortest call there is; the caller waits for its result
        _case("f32-single-spec", "c0", "spec", 1, 7, 384, 2, stats=True),
        # fp32, a ragged batch and a horizon that is no whole number of patches
        _case("f32-ragged-spec", "c0", "spec", 37, 20, 1000, 3),
        # interactive forecast of one series with the 25 M model
        _case("single-spec", "c1", "spec", 1, 30, 720, 4, stats=True),
        # a batch of channels, longer horizon
        _case("channels-spec", "c1", "spec", 32, 30, 1440, 4),
        # a data frame of eleven series in host memory, plain decoding
        _case("frame-target-host", "c1", "target", 11, 29, 700, host=True),
        # wide multivariate sets on the 300 M model: speculative and plain, full and odd batch
        _case("wide-spec", "c2", "spec", 256, 30, 720, 4),
        _case("wide-ragged-target", "c2", "target", 93, 27, 720),
        # scoring windows with the 300 M model
        _case("wide-score", "c2", "forward", 200, 30),
        # a thousand short series
        _case("many-short-spec", "c3", "spec", 1024, 7, 1440, 4),
        # long context and horizon on the 500 M model
        _case("long-spec", "c4", "spec", 64, 256, 2048, 8),
        _case("long-target", "c4", "target", 64, 256, 2048),
        # point tokens
        _case("points-spec", "c5", "spec", 16, 12, 384, 3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(sorted(FAMILIES))
    F = FAMILIES[family]
    op = rng.choice(["spec", "spec", "target", "forward"])
    B = _log_int(rng, 1, F["B"])
    ctx = _log_int(rng, max(2, F["ctx"] // 8), F["ctx"])
    if op == "forward":
        return _case(None, family, op, B, ctx)
    H = rng.randint(max(1, F["T"] * F["P"] // 4), F["T"] * F["P"])
    K = _log_int(rng, 1, F["K"]) if op == "spec" else 0
    host = rng.random() < 0.25
    return _case(None, family, op, B, ctx, H, K, host=host, stats=not host and rng.random() < 0.25)


# ------------------------------------------------------------------------------------------ weights and series
def _tensors(a, P, P_in):
    d, f = a.d_model, a.d_ff
    yield -1, "W_emb", (d, P_in or P)
    for l in range(a.n_layers):
        for n, s in (("g1", (d,)), ("Wq", (d, d)), ("Wk", (d, d)), ("Wv", (d, d)), ("Wo", (d, d)), ("g2", (d,)),
                     ("W1", (f, d)), ("W2", (d, f))):
            yield l, n, s
    yield -1, "g_f", (d,)
    yield -1, "W_head", (P, d)


def _persistence(W_emb, W_head, P, gen):
    """Embedding with orthogonal columns and the head that reads them back: after the final norm the prediction is
    the last token's direction, repeated over the patch.  (One point's direction is its sign: there the head keeps a
    part that reads everything else.)"""
    d, p = W_emb.shape
    Q = torch.linalg.qr(torch.randn(d, p, device="cuda", generator=gen)).Q
    W_emb.copy_(Q * math.sqrt(d / p))
    W_head.mul_(POINT_HEAD if p < P else 0.0).add_((Q * math.sqrt(p / d)).T.repeat(P // p, 1))


def _model(arch, F, gen, damp):
    """Weight tensors by (layer, name), fp32.  damp(layer) scales Wo and W2 of a layer."""
    w = {}
    for l, n, s in _tensors(arch, F["P"], F["P_in"]):
        if len(s) == 1:
            w[l, n] = torch.ones(s, device="cuda")
            continue
        t = torch.randn(s, device="cuda", generator=gen) * math.sqrt(2.0 / sum(s))
        w[l, n] = t * damp(l) if n in ("Wo", "W2") else t
    return w


def _pack(w, arch, F):
    """The device blob that the library reads (layout from the library's own offsets)."""
    P, P_in, dt = F["P"], F["P_in"], F["dtype"]
    blob = torch.zeros(tsfm.tsfm_weights_bytes_io(arch, P_in, P, dt), dtype=torch.uint8, device="cuda")
    head = torch.tensor([0x4D465354, 1, tsfm.TSFM_BF16 if dt == "bf16" else tsfm.TSFM_F32, arch.n_layers, arch.d_model,
                         arch.n_heads, arch.d_ff, P, P_in], dtype=torch.int32)
    blob[:36] = head.view(torch.uint8).cuda()
    for (l, n), t in w.items():
        t = t.to(torch.bfloat16) if dt == "bf16" and t.dim() == 2 else t
        raw = t.contiguous().view(-1).view(torch.uint8)
        off = tsfm.tsfm_weights_offset_io(arch, P_in, P, dt, l, n)
        blob[off:off + raw.numel()] = raw
    return blob


def _weights(case, gen):
    """Weight tensors of target and draft (None: the draft is the target's first layers)."""
    F = FAMILIES[case["family"]]
    ta, da = tsfm.tsfm_arch(*F["target"]), tsfm.tsfm_arch(*F["draft"])
    tracking = case["op"] == "spec" and F["dtype"] == "bf16"
    damp = lambda l: 1.0  # noqa: E731
    if tracking and F["mode"] == "layer_skip":
        damp = lambda l: 1.0 if l < da.n_layers else LATE_LAYERS  # noqa: E731
    elif tracking and F["mode"] == "separate":
        damp = lambda l: POINT_CORRECTION if F["P_in"] else CORRECTION  # noqa: E731
    t = _model(ta, F, gen, damp)
    if F["mode"] == "layer_skip":
        return t, None
    if F["mode"] == "perturbed":
        d = {k: v if v.dim() == 1 else v + PERTURBATION * v.std() * torch.randn(v.shape, device="cuda", generator=gen)
             for k, v in t.items()}
    else:
        d = _model(da, F, gen, damp)
        if tracking:
            for w in (t, d):
                _persistence(w[-1, "W_emb"], w[-1, "W_head"], F["P"], gen)
    return t, d


def _models(case, gen):
    F = FAMILIES[case["family"]]
    ta, da = tsfm.tsfm_arch(*F["target"]), tsfm.tsfm_arch(*F["draft"])
    t, d = _weights(case, gen)
    return ta, da, _pack(t, ta, F), None if d is None else _pack(d, da, F)


def _series(B, n, gen):
    """Seasonal + trend + AR(1) noise + level shifts, z-normalised per series."""
    rnd = lambda *s: torch.rand(s, device="cuda", generator=gen)  # noqa: E731
    t = torch.arange(n, device="cuda", dtype=torch.float32)
    period = 12.0 * 2.0 ** torch.floor(3 * rnd(B, 1))
    y = torch.sin(2 * math.pi * t / period) + 0.5 * torch.sin(2 * math.pi * t / 168) + (0.04 * rnd(B, 1) - 0.02) * t
    ar = 0.8 ** torch.arange(63, -1, -1, device="cuda", dtype=torch.float32)
    noise = 0.1 * torch.randn(B, 1, n + 63, device="cuda", generator=gen)
    y = y + torch.nn.functional.conv1d(noise, ar.view(1, 1, -1)).squeeze(1)
    y = y + torch.cumsum((rnd(B, n) < 1 / 500) * 2.0 * torch.randn(B, n, device="cuda", generator=gen), 1)
    return ((y - y.mean(1, keepdim=True)) / y.std(1, keepdim=True)).contiguous()


class _State:
    """What a program that forecasts keeps: weights, the decoder handle, its series and a result buffer."""

    def __init__(self, case, seed):
        F = FAMILIES[case["family"]]
        gen = torch.Generator(device="cuda").manual_seed(seed)
        self.case, self.F, self.seed = case, F, seed
        ta, da, self.target, self.draft = _models(case, gen)
        P, B = F["P"], case["B"]
        P_in = F["P_in"] or P
        self.n_tok = case["ctx"] * P // P_in
        cfg = tsfm.tsfm_cfg()
        cfg.target, cfg.draft, cfg.patch_len, cfg.patch_in = ta, da, P, F["P_in"]
        cfg.dtype = tsfm.TSFM_BF16 if F["dtype"] == "bf16" else tsfm.TSFM_F32
        cfg.draft_mode = tsfm.TSFM_DRAFT_LAYER_SKIP if self.draft is None else tsfm.TSFM_DRAFT_SEPARATE
        cfg.max_batch, cfg.max_ctx_tokens = B, self.n_tok
        cfg.max_horizon_patches, cfg.max_K = max(1, -(-case["H"] // P)), max(1, case["K"])
        cfg.rms_eps, cfg.norm_eps, cfg.rope_base = 1e-6, 1e-5, 1e4
        cfg.stream = torch.cuda.current_stream().cuda_stream
        s = _series(B, case["ctx"] * P, gen)
        if case["op"] == "forward":
            self.x = s.view(B, self.n_tok, P_in)
            self.out = torch.empty(B, self.n_tok, P, device="cuda")
        else:
            self.x, self.out = s, torch.empty(B, case["H"], device="cuda")
        if case["host"]:
            self.x, self.out = self.x.cpu().numpy(), self.out.cpu().numpy()
        self.handle = tsfm.tsfm_spec_create(self.target, self.draft, cfg)

    def __del__(self):
        if getattr(self, "handle", None):
            tsfm.tsfm_spec_destroy(self.handle)
            self.handle = None


def prepare(case, seed):
    return _State(case, seed)


def run(st):
    c = st.case
    n = c["ctx"] * st.F["P"]
    stats = tsfm.tsfm_stats() if c["stats"] else None
    if c["op"] == "forward":
        tsfm.tsfm_model_forward(st.handle, 0, st.x, c["B"], st.n_tok, st.out)
    elif c["op"] == "target":
        f = tsfm.tsfm_target_only_forecast_host if c["host"] else tsfm.tsfm_target_only_forecast
        f(st.handle, st.x, c["B"], n, c["H"], st.out, stats)
    else:
        f = tsfm.tsfm_spec_forecast_host if c["host"] else tsfm.tsfm_spec_forecast
        f(st.handle, st.x, c["B"], n, c["H"], c["K"], st.F["tau"], st.seed, st.out, stats)
    return st.out


# ------------------------------------------------------------------------------------------ the same in 64 bits
def _rotate(t, cos, sin):
    a, b = t.chunk(2, -1)
    return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)


def _norm(x, g):
    return g * x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-6)


class _Plain:
    """Pre-norm decoder with rotary positions and a key/value cache, plain torch in 64 bits."""

    def __init__(self, w, arch, B, cap):
        self.w, (self.L, d, self.heads, _) = w, arch
        self.dh, self.pos = d // self.heads, 0
        angle = torch.arange(cap, device="cuda", dtype=torch.float64)[:, None] * 1e4 ** (
            -2.0 * torch.arange(self.dh // 2, device="cuda", dtype=torch.float64) / self.dh)
        self.cos, self.sin = angle.cos(), angle.sin()
        self.kv = torch.empty(self.L, 2, B, self.heads, cap, self.dh, device="cuda", dtype=torch.float64)

    def __call__(self, z):
        """z [B, n, values per token] behind what was given before -> next-patch means [B, n, P]."""
        w, (B, n, _), p = self.w, z.shape, self.pos
        split = lambda t: t.view(B, n, self.heads, self.dh).transpose(1, 2)  # noqa: E731
        cos, sin = self.cos[p:p + n], self.sin[p:p + n]
        mask = torch.ones(n, p + n, device="cuda", dtype=torch.bool).tril(p)
        x = z @ w[-1, "W_emb"].T
        for l in range(self.L):
            a = _norm(x, w[l, "g1"])
            K, V = self.kv[l, 0, :, :, :p + n], self.kv[l, 1, :, :, :p + n]
            K[:, :, p:] = _rotate(split(a @ w[l, "Wk"].T), cos, sin)
            V[:, :, p:] = split(a @ w[l, "Wv"].T)
            s = _rotate(split(a @ w[l, "Wq"].T), cos, sin) @ K.transpose(2, 3) / math.sqrt(self.dh)
            s = s.masked_fill(~mask, -math.inf).softmax(-1)
            x = x + (s @ V).transpose(1, 2).reshape(B, n, -1) @ w[l, "Wo"].T
            h = torch.nn.functional.gelu(_norm(x, w[l, "g2"]) @ w[l, "W1"].T)
            x = x + h @ w[l, "W2"].T
        self.pos = p + n
        return _norm(x, w[-1, "g_f"]) @ w[-1, "W_head"].T


@torch.no_grad()
def exact(case, seed):
    """Scoring and plain forecasts.  A speculative forecast has none: a decision that falls within rounding of its
    threshold has two valid outcomes."""
    if case["op"] == "spec":
        return None
    F = FAMILIES[case["family"]]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    w, _ = _weights(case, gen)
    w = {k: (v.to(torch.bfloat16) if F["dtype"] == "bf16" and v.dim() == 2 else v).double() for k, v in w.items()}
    B, P = case["B"], F["P"]
    P_in = F["P_in"] or P
    s = _series(B, case["ctx"] * P, gen).double()
    T = -(-case["H"] // P)
    model = _Plain(w, F["target"], B, (case["ctx"] + T) * P // P_in)
    if case["op"] == "forward":
        return model(s.view(B, -1, P_in))
    mean, sd = s.mean(1, keepdim=True), (s.var(1, keepdim=True, unbiased=False) + 1e-5).sqrt()
    z, patches = (s - mean) / sd, []
    for _ in range(T):
        z = model(z.view(B, -1, P_in))[:, -1]
        patches.append(z)
    out = (torch.cat(patches, 1) * sd + mean)[:, :case["H"]].contiguous()
    return out.cpu().numpy() if case["host"] else out


# ------------------------------------------------------------------------------------------ what a pass needs at least
L2_BYTES = 126 << 20


def work(case):
    """Contractions and attention of every token that has to be computed, and for every pass of a model that has to
    follow another one (a decoded patch, a drafted patch, a verification) its weights and cached keys and values -- once
    in all where they stay in the L2 cache between such passes.  A speculative forecast is counted with every proposal
    accepted."""
    F = FAMILIES[case["family"]]
    e, P = (2 if F["dtype"] == "bf16" else 4), F["P"]
    tpp = P // (F["P_in"] or P)                       # tokens per patch
    B, N = case["B"], case["ctx"] * tpp
    T = -(-case["H"] // P)
    total = {"bytes": 0.0, "flops": 0.0}

    def model(arch, first, passes, q, heads):
        """`first` tokens at once (no head unless heads), then `passes` passes of q tokens each."""
        L, d, _, f = arch
        mats = L * (4 * d * d + 2 * d * f)
        tokens = first + passes * q
        keys = first * (first + 1) / 2 + sum(q * (first + i * q + (q + 1) / 2) for i in range(passes))
        total["flops"] += B * (2.0 * mats * tokens + 4.0 * L * d * keys + 2.0 * d * (P // tpp) * tokens + 2.0 * d * P * heads)
        weights = e * (mats + d * P + d * P // tpp)
        kv = 2.0 * e * B * L * d * (first + passes * q / 2)
        stream = max(1, passes)
        total["bytes"] += weights * (stream if weights > L2_BYTES else 1)
        total["bytes"] += kv * (passes if kv > L2_BYTES else min(passes, 1)) + 2.0 * e * B * L * d * tokens

    if case["op"] == "forward":
        model(F["target"], N, 0, 0, N)
        total["bytes"] += 4.0 * B * (case["ctx"] * P + N * P)
        return total
    total["bytes"] += 4.0 * B * (case["ctx"] * P + case["H"])
    if case["op"] == "target":
        model(F["target"], N - tpp, T, tpp, T)
    else:
        K, rounds = case["K"], -(-T // (case["K"] + 1))
        model(F["target"], N - tpp, rounds, (K + 1) * tpp, rounds * (K + 1))
        model(F["draft"], N - tpp, rounds * K, tpp, rounds * K)
    return total


def tolerance(case):
    """Measured by running the bf16 contractions with their sums in another order (FMA kernels instead of the tensor
    cores): plain forecasts and scoring differ by 2.5e-3 to 6e-3.  A speculative forecast differs as little until a
    decision falls within rounding of its threshold: from there on that series takes its other, equally valid branch,
    which with these draft / target pairs moves a patch by about a tenth of its size (1.5e-2 over a batch, single
    values by up to 0.42 of the rms).  fp32 sums in another order: a few 1e-6."""
    if FAMILIES[case["family"]]["dtype"] == "f32":
        return {"rel": 1e-5}
    if case["op"] == "spec":
        return {"rel": 3e-2, "max": 0.99}
    return {"rel": 2e-2, "max": 0.2}
