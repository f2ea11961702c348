"""Performance cases: the work that a user of the library has it do.

Six ways in, each through the public binding (`paper_2608_09231_gb300.bag`):

  sample     `Context.run`: all T steps of one sample under Algorithm 2
  steps      `Context.step`: the same sample step by step, as a program with its own loop
  block      `Context.forward_block`: one block of the stack on a residual stream
  attention  `Context.attention_f16`: multi-head attention of given q, k, V^T
  mlp        `Context.gemm_bf16`: a projection with bias and GELU
  norm       `Context.ln_mod`: LayerNorm with adaLN modulation
  signal     `rel_l1_noalloc` / `Context.rel_l1`: relative L1 change of two tensors

`exact` restates each of them in float64 with plain torch (its own weight generator, the
published SplitMix64, and its own network), at sizes where that takes seconds.
"""

import math

import numpy as np
import torch

from paper_2608_09231_gb300 import bag

DEV = "cuda"
PATCH = 64          # latent channels per image token
TEMB = 256          # width of the sinusoidal timestep embedding
MODEL_OPS = ("sample", "steps", "block")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _model(op, kind, hidden, heads, mlp, blocks, grid, n_txt, T, B, dtype="bf16", **more):
    """A case on a backbone; blocks = (n_double, n_single, n_wan)."""
    c = dict(op=op, kind=kind, hidden=hidden, heads=heads, mlp=mlp, n_double=blocks[0],
             n_single=blocks[1], n_wan=blocks[2], frames=grid[0], rows=grid[1], cols=grid[2],
             n_txt=n_txt, T=T, B=B, dtype=dtype, guidance=0.0, qk_norm=False, gate_kind="mlp3",
             sampler="euler", shift=1.0, observable="modulated")
    c.update(more)
    return c


def listed():
    return [
        # the signal reduction inside another framework's loop, on the smallest backbone's
        # tokens (256 x 256, fp32): a call that is all latency
        dict(name="signal_tiny_f32", op="signal", rows=256, cols=256, dtype="f32", noalloc=True),
        # the same on the FLUX-shaped observable (4096 tokens x 3072, bf16)
        dict(name="signal_flux_bf16", op="signal", rows=4096, cols=3072, dtype="bf16", noalloc=False),
        # LayerNorm + modulation of the FLUX-shaped joint sequence (512 + 4096 tokens)
        dict(name="norm_flux_joint", op="norm", rows=4608, cols=3072),
        # MLP up-projection with GELU of a ragged text / low-resolution image stream
        dict(name="mlp_up_ragged", op="mlp", M=1373, N=12288, K=3072),
        # joint attention at the Qwen-Image-shaped token count (83 x 83 image + 256 text)
        dict(name="attention_qwen", op="attention", nq=7145, nk=7145, heads=24),
        # toy-scale fp32 backbone, one rollout of the schedule search: latency and launches
        dict(name="sample_tiny_f32",
             **_model("sample", "single", 256, 4, 1024, (0, 2, 0), (1, 16, 16), 32, 10, 5, "f32")),
        # a reduced FLUX-shaped backbone with everything the FLUX runs use: guidance, QK-norm,
        # the six-input gate, the post-patch-embedding observable
        dict(name="sample_flux_small_guided",
             **_model("sample", "mmdit", 512, 4, 2048, (2, 2, 0), (1, 18, 21), 77, 10, 5,
                      guidance=4.0, qk_norm=True, gate_kind="flux6", observable="embedded")),
        # a reduced Wan-shaped backbone: 3-D grid, cross-attention, UniPC on a shifted grid
        dict(name="sample_wan_small",
             **_model("sample", "wan", 512, 4, 1536, (0, 0, 2), (3, 10, 13), 70, 10, 4,
                      gate_kind="wan6", sampler="unipc", shift=5.0)),
        # one FLUX-shaped single-stream block driven step by step at the lowest budget of
        # the paper's FLUX runs (10 of 50): four steps in five take the reuse path
        dict(name="steps_flux_block",
             **_model("steps", "single", 3072, 24, 12288, (0, 1, 0), (1, 64, 64), 512, 50, 10)),
        # one FLUX-shaped double-stream block, QK-norm on
        dict(name="block_flux_double",
             **_model("block", "mmdit", 3072, 24, 12288, (1, 0, 0), (1, 64, 64), 512, 4, 2,
                      qk_norm=True)),
        # one Wan2.1-14B-shaped block on an 81-frame 480x832 video (32,760 tokens)
        dict(name="block_wan",
             **_model("block", "wan", 5120, 40, 13824, (0, 0, 1), (21, 30, 52), 512, 4, 2)),
        # the headline: a FLUX-shaped sample, 20 full evaluations in 50 steps
        dict(name="sample_flux",
             **_model("sample", "mmdit", 3072, 24, 12288, (19, 38, 0), (1, 64, 64), 512, 50, 20)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["signal", "norm", "mlp", "attention", "sample", "sample", "steps", "block"])
    if op == "signal":
        cols = rng.choice([256, 512, 1024, 1536, 2048, 3072, 4096, 5120, _log_int(rng, 64, 5120)])
        return dict(op=op, rows=_log_int(rng, 64, 32760), cols=cols, dtype=rng.choice(["f32", "bf16"]),
                    noalloc=rng.random() < 0.5)
    if op == "norm":
        return dict(op=op, rows=_log_int(rng, 64, 32760),
                    cols=rng.choice([256, 512, 1024, 1536, 2048, 3072, 4096, 5120, 4 * _log_int(rng, 64, 1536)]))
    if op == "mlp":
        K = 64 * _log_int(rng, 4, 80)
        return dict(op=op, M=_log_int(rng, 32, 8192), N=64 * _log_int(rng, 4, 216), K=K)
    if op == "attention":
        nq = _log_int(rng, 64, 9000)
        return dict(op=op, nq=nq, nk=rng.choice([nq, nq, 512, _log_int(rng, 32, 2048)]),
                    heads=rng.choice([2, 4, 8, 16, 24, 40]))
    if op == "sample" and rng.random() < 0.35:
        # toy-scale fp32 backbones
        dh = rng.choice([64, 64, 128])
        heads = rng.choice([2, 4, 6])
        T = rng.randint(6, 14)
        return _model(op, "single", dh * heads, heads, 4 * dh * heads, (0, rng.randint(1, 3), 0),
                      (1, rng.randint(6, 20), rng.randint(6, 20)), rng.randint(5, 48), T,
                      rng.randint(2, T - 1), "f32", gate_kind=rng.choice(["mlp3", "flux6", "wan6"]))
    kind = rng.choice(["single", "mmdit", "wan"])
    T = rng.randint(6, 28)
    B = rng.randint(2, max(2, T // 2))
    more = {}
    if op == "block":
        T, B = 4, 2
        heads = rng.choice([4, 8, 16, 24])
        tokens = _log_int(rng, 200, 8000)
        blocks = {"single": (0, 1, 0), "mmdit": (1, 0, 0), "wan": (0, 0, 1)}[kind]
    elif op == "steps":
        heads = rng.choice([4, 8, 24])
        tokens = _log_int(rng, 200, 4096)
        blocks = {"single": (0, 1, 0), "mmdit": (1, 0, 0), "wan": (0, 0, 1)}[kind]
    else:
        heads = rng.choice([4, 8, 12])
        tokens = _log_int(rng, 150, 1600)
        n = rng.randint(1, 3)
        blocks = {"single": (0, n, 0), "mmdit": (n, rng.randint(0, 2), 0), "wan": (0, 0, n)}[kind]
        more["guidance"] = rng.choice([0.0, 0.0, 4.0])
    frames = rng.randint(2, 5) if kind == "wan" else 1
    side = math.sqrt(tokens / frames)
    rows = max(3, int(round(side * rng.uniform(0.7, 1.3))))
    cols = max(3, int(round(tokens / frames / rows)))
    hidden = 128 * heads
    more["qk_norm"] = kind != "wan" and rng.random() < 0.5
    more["gate_kind"] = rng.choice(["mlp3", "flux6", "wan6"])
    more["observable"] = rng.choice(["modulated", "embedded"])
    if kind == "wan":
        more.update(sampler="unipc", shift=5.0)
    return _model(op, kind, hidden, heads, hidden * rng.choice([3, 4]), blocks, (frames, rows, cols),
                  rng.randint(20, 512), T, B, **more)


# ---------------------------------------------------------------------------
# inputs and state
# ---------------------------------------------------------------------------
GATE_SHAPES = {  # (out, in) of every layer in storage order
    "mlp3": [(16, 3), (1, 16)],
    "flux6": [(8, 6), (8, 8), (32, 8), (1, 32)],
    "wan6": [(8, 3), (8, 8), (8, 3), (8, 8), (32, 16), (1, 32)],
}


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32).to(dtype)


def _axes(case):
    dh = case["hidden"] // case["heads"]
    if case["kind"] == "wan":
        return (44, 42, 42)
    return (0, 32, 32) if dh == 64 else (16, 56, 56)


def _config(case, seed):
    return dict(kind=case["kind"], hidden=case["hidden"], heads=case["heads"], mlp=case["mlp"],
                n_double=case["n_double"], n_single=case["n_single"], n_wan=case["n_wan"],
                grid=(case["frames"], case["rows"], case["cols"]), n_txt=case["n_txt"],
                patch_ch=PATCH, rope_axes=_axes(case), dtype=case["dtype"],
                weight_seed=int(seed) & 0x7FFFFFFF, gate_seed=int(seed) & 0x7FFFFFFF,
                guidance=case["guidance"] or None, qk_norm=case["qk_norm"],
                gate_kind=case["gate_kind"], sampler=case["sampler"], shift=case["shift"],
                observable=case["observable"], T=case["T"], budgets=(case["B"],))


def _gate(case, seed):
    """A gate of the case's kind, as a trained one is loaded: parameters (Xavier-uniform),
    z-score mean and standard deviation of its inputs."""
    r = np.random.RandomState(int(seed) & 0x7FFFFFFF)
    layers = []
    for out, inn in GATE_SHAPES[case["gate_kind"]]:
        a = math.sqrt(6.0 / (inn + out))
        layers.append((r.uniform(-a, a, (out, inn)).astype(np.float32),
                       r.uniform(-0.1, 0.1, out).astype(np.float32)))
    if case["gate_kind"] == "mlp3":
        mu, sd = [0.5, 0.5, 0.3], [0.3, 0.3, 0.25]
    else:
        mu, sd = [0.4, 0.5, 0.4, 2.0, 0.3, 0.1], [0.2, 0.3, 0.2, 1.5, 0.25, 0.1]
    return layers, np.float32(mu), np.float32(sd)


def _sample_inputs(case, seed):
    g = _gen(seed)
    ni = case["frames"] * case["rows"] * case["cols"]
    d, nx = case["hidden"], case["n_txt"]
    tt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    s = dict(x0=_randn(g, ni, PATCH), txt=_randn(g, nx, d, dtype=tt), pooled=_randn(g, d))
    if case["guidance"]:
        s.update(txt_u=_randn(g, nx, d, dtype=tt), pooled_u=_randn(g, d))
    return s


def _block_input(case, seed):
    g = _gen(int(seed) + 1)
    ni = case["frames"] * case["rows"] * case["cols"]
    n = ni if case["kind"] == "wan" else ni + case["n_txt"]
    return _randn(g, n, case["hidden"])


def _op_inputs(case, seed):
    g = _gen(seed)
    op = case["op"]
    if op == "signal":
        tt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        b = _randn(g, case["rows"], case["cols"])
        a = b + 0.2 * _randn(g, case["rows"], case["cols"])   # a later step's observable
        return dict(a=a.to(tt), b=b.to(tt))
    if op == "norm":
        # a residual stream: a common offset and rows of different size
        x = _randn(g, case["rows"], case["cols"]) * (0.5 + torch.rand(case["rows"], 1, generator=g, device=DEV))
        return dict(x=x + 0.3, shift=0.3 * _randn(g, case["cols"]), scale=0.3 * _randn(g, case["cols"]))
    if op == "mlp":
        return dict(A=_randn(g, case["M"], case["K"], dtype=torch.bfloat16),
                    W=(0.02 * _randn(g, case["N"], case["K"])).to(torch.bfloat16),
                    bias=0.02 * _randn(g, case["N"]))
    H, nq, nk = case["heads"], case["nq"], case["nk"]
    vpad = (nk + 127) // 128 * 128
    vt = torch.zeros(H, 128, vpad, device=DEV, dtype=torch.float16)
    q, k = _randn(g, nq, H * 128, dtype=torch.float16), _randn(g, nk, H * 128, dtype=torch.float16)
    vt[:, :, :nk] = _randn(g, H, 128, nk, dtype=torch.float16)
    return dict(q=q, k=k, vt=vt, vpad=vpad)


def _op_context(seed):
    """A small context: the single-operation calls need one for its stream and errors."""
    return bag.create("tiny", weight_seed=int(seed) & 0x7FFFFFFF)


def prepare(case, seed):
    op = case["op"]
    if op in MODEL_OPS:
        ctx = bag.create(_config(case, seed), T=case["T"], B=case["B"])
        layers, mu, sd = _gate(case, seed)
        ctx.load_gate(np.concatenate([np.concatenate([w.ravel(), b]) for w, b in layers]), mu, sd)
        s = dict(case=case, ctx=ctx, **_sample_inputs(case, seed))
        s["cond"] = [s["txt"], s["pooled"]]
        s["cond_u"] = [s.get("txt_u"), s.get("pooled_u")]
        if op == "block":
            s["h0"] = _block_input(case, seed)
            s["h"] = torch.empty_like(s["h0"])
            ctx.prepare(*s["cond"], *s["cond_u"])
        else:
            s["x"] = torch.empty_like(s["x0"])
            s["flags"] = torch.zeros(case["T"], device=DEV, dtype=torch.int32)
        return s
    s = dict(case=case, **_op_inputs(case, seed))
    if op == "signal":
        s["out"] = torch.empty(3, device=DEV)
        if not case["noalloc"]:
            s["ctx"] = _op_context(seed)
            s["scratch"] = torch.empty(2 * case["rows"], device=DEV)
        return s
    s["ctx"] = _op_context(seed)
    if op == "norm":
        s["y"] = torch.empty(case["rows"], case["cols"], device=DEV, dtype=torch.bfloat16)
    elif op == "mlp":
        s["C"] = torch.empty(case["M"], case["N"], device=DEV)
    else:
        s["o"] = torch.empty(case["nq"], case["heads"] * 128, device=DEV, dtype=torch.bfloat16)
    return s


def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "sample":
        s["x"].copy_(s["x0"])
        s["ctx"].reset()
        mask, log, _ = s["ctx"].run(s["x"], *s["cond"], *s["cond_u"])
        return {"latent": s["x"], "mask": mask, "log": log}
    if op == "steps":
        s["x"].copy_(s["x0"])
        s["ctx"].reset()
        for t in range(case["T"]):
            s["ctx"].step(s["x"], t, *s["cond"], s["x"], s["flags"][t:t + 1], *s["cond_u"])
        return {"latent": s["x"], "flags": s["flags"]}
    if op == "block":
        s["h"].copy_(s["h0"])
        s["ctx"].forward_block(0, case["T"] // 2, s["h"])
        return s["h"]
    if op == "attention":
        s["ctx"].attention_f16(s["q"], s["k"], s["vt"], s["o"], case["nq"], case["nk"], case["heads"],
                               128, s["vpad"])
        return s["o"]
    if op == "mlp":
        s["ctx"].gemm_bf16(s["A"], s["W"], s["bias"], s["C"], case["M"], case["N"], case["K"], epilogue=1)
        return s["C"]
    if op == "norm":
        s["ctx"].ln_mod(s["x"], s["shift"], s["scale"], s["y"], case["rows"], case["cols"])
        return s["y"]
    if case["noalloc"]:
        bag.rel_l1_noalloc(s["a"], s["b"], case["rows"], case["cols"], s["out"])
    else:
        s["ctx"].rel_l1(s["a"], s["b"], case["rows"], case["cols"], s["scratch"], s["out"])
    return s["out"]


# ---------------------------------------------------------------------------
# algorithmic work and tolerances
# ---------------------------------------------------------------------------
def _block_types(case):
    return ["wan"] * case["n_wan"] + ["double"] * case["n_double"] + ["single"] * case["n_single"]


def _block_work(case, kind):
    """(flops, weight elements) of one block on one branch."""
    d, F, nx = case["hidden"], case["mlp"], case["n_txt"]
    ni = case["frames"] * case["rows"] * case["cols"]
    N = ni + nx
    if kind == "single":
        w = d * (3 * d + F) + d * (d + F)
        return 2.0 * N * w + 4.0 * N * N * d, w
    if kind == "double":
        w = 4 * d * d + 2 * d * F
        return 2.0 * N * w + 4.0 * N * N * d, 2 * w
    w = 6 * d * d + 2 * d * F
    return 2.0 * ni * w + 4.0 * nx * d * d + 4.0 * ni * ni * d + 4.0 * ni * nx * d, w + 2 * d * d


def work(case):
    op = case["op"]
    if op == "signal":
        n, es = case["rows"] * case["cols"], 4 if case["dtype"] == "f32" else 2
        return {"bytes": 2 * n * es + 12, "flops": 5 * n}
    if op == "norm":
        n = case["rows"] * case["cols"]
        return {"bytes": 6 * n + 8 * case["cols"], "flops": 8 * n}
    if op == "mlp":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * (M + N) * K + 4 * N + 4 * M * N, "flops": 2 * M * N * K}
    if op == "attention":
        d = 128 * case["heads"]
        return {"bytes": 4 * d * (case["nq"] + case["nk"]), "flops": 4 * case["nq"] * case["nk"] * d}
    es = 4 if case["dtype"] == "f32" else 2
    d, T, B = case["hidden"], case["T"], case["B"]
    ni = case["frames"] * case["rows"] * case["cols"]
    br = 2 if case["guidance"] else 1
    blocks = [_block_work(case, k) for k in _block_types(case)]
    flops, weights = sum(b[0] for b in blocks) * br, sum(b[1] for b in blocks)
    if op == "block":
        n = ni if case["kind"] == "wan" else ni + case["n_txt"]
        return {"bytes": weights * es + 8 * n * d, "flops": flops}
    # once a sample: the conditioning projections; every step: patch embedding, signal (the
    # observable against its two references, and its new value), final layer; a full step:
    # the stack's weights and the new residual; a reused one: the cached residual
    n_mod = sum({"single": 3, "double": 12, "wan": 0}[k] for k in _block_types(case)) * d + 2 * d
    n_mod += 6 * d if case["kind"] == "wan" else 0
    obs = 4 if case["observable"] == "embedded" else es
    step = 3.0 * ni * d * obs + 8.0 * ni * PATCH + 2.0 * d * PATCH * es
    bytes_ = n_mod * d * es + T * step + B * weights * es + T * br * 4.0 * ni * d
    flops_ = 2.0 * T * n_mod * d * br + T * (1 + br) * 2.0 * ni * d * PATCH + B * flops
    return {"bytes": bytes_, "flops": flops_}


def tolerance(case):
    """About four times the error against `exact` (bf16 outputs: their rounding, 1.7e-3;
    whole samples: 16-bit projection and attention operands through every layer and step;
    fp32 projections: sums over up to 5120 products)."""
    op = case["op"]
    if op == "signal":
        return {"rel": 2e-6}
    if op == "norm":
        return {"rel": 7e-3, "max": 0.03}
    if op == "mlp":
        return {"rel": 1.5e-5}
    if op == "attention":
        return {"rel": 7e-3, "max": 0.03}
    if case["dtype"] == "f32":
        return {"rel": 5e-6}
    if op == "block":
        return {"rel": 8e-3, "max": 0.06}
    return {"rel": 1e-2, "max": 0.1}


# ---------------------------------------------------------------------------
# the same in float64
# ---------------------------------------------------------------------------
def _i64(u):
    return u - (1 << 64) if u >= 1 << 63 else u


def _mix_int(z):
    z &= (1 << 64) - 1
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & ((1 << 64) - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & ((1 << 64) - 1)
    return z ^ (z >> 31)


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _normal(seed, key, n, std, chunk=1 << 25):
    """The seeded generator (SplitMix64 stream of a tensor key; the four 16-bit chunks of
    an output summed and centred), as fp32 values."""
    golden = 0x9E3779B97F4A7C15
    start = _mix_int((seed * golden) ^ _mix_int(key))
    out = torch.empty(n, device=DEV)
    c32 = torch.tensor(np.float32(std * math.sqrt(3.0) / 65536.0), device=DEV)
    for a in range(0, n, chunk):
        i = torch.arange(a + 1, min(n, a + chunk) + 1, device=DEV, dtype=torch.int64)
        z = i * _i64(golden) + _i64(start)
        z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
        z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
        z = z ^ _shr(z, 31)
        q = sum((_shr(z, s) if s else z) & 0xFFFF for s in (0, 16, 32, 48)) - 131070
        out[a:a + chunk] = q.to(torch.float32) * c32
    return out


class _Net:
    """The backbone of a case in float64: weights from the seed, blocks, embedding, head."""

    def __init__(self, case, seed):
        self.c, self.seed = case, int(seed) & 0x7FFFFFFF
        self.d, self.H, self.F, self.nx = case["hidden"], case["heads"], case["mlp"], case["n_txt"]
        self.dh = self.d // self.H
        self.wan = case["kind"] == "wan"
        d = self.d
        ids = [("pe", d, PATCH), ("t1", d, TEMB), ("t2", d, d), ("fmod", 2 * d, d), ("fin", PATCH, d)]
        if self.wan:
            ids.append(("tproj", 6 * d, d))
        self.G = {n: self._linear(0, 2 * i, o, k) for i, (n, o, k) in enumerate(ids)}
        self.blocks = [(k, self._block(1 + i, k)) for i, k in enumerate(_block_types(case))]
        self.angles = self._angles()

    def _tensor(self, slot, tid, shape, round16=False, offset=0.0):
        v = _normal(self.seed, slot * 256 + tid, int(np.prod(shape)), 0.02).reshape(shape)
        if offset:
            v = v + offset
        if round16 and self.c["dtype"] == "bf16":
            v = v.to(torch.bfloat16)
        return v.double()

    def _linear(self, slot, tid, out, inn):
        return self._tensor(slot, tid, (out, inn), True), self._tensor(slot, tid + 1, (out,))

    def _block(self, slot, kind):
        d, F = self.d, self.F
        L = lambda tid, o, i: self._linear(slot, tid, o, i)   # noqa: E731
        norm = lambda tid: self._tensor(slot, tid, (self.dh,), offset=1.0)   # noqa: E731
        if kind == "single":
            w = {"mod": L(0, 3 * d, d), "lin1": L(2, 3 * d + F, d), "lin2": L(4, d, d + F)}
            if self.c["qk_norm"]:
                w["norm"] = (norm(6), norm(7))
            return w
        if kind == "double":
            w = {}
            for i, s in enumerate(("img", "txt")):
                for j, (n, o, k) in enumerate((("mod", 6 * d, d), ("qkv", 3 * d, d), ("proj", d, d),
                                               ("up", F, d), ("down", d, F))):
                    w[s + n] = L(10 * i + 2 * j, o, k)
                if self.c["qk_norm"]:
                    w[s + "norm"] = (norm(20 + 2 * i), norm(21 + 2 * i))
            return w
        w = {"tab": self._tensor(slot, 0, (6 * d,))}
        for j, (n, o, k) in enumerate((("sa_qkv", 3 * d, d), ("sa_o", d, d), ("ca_q", d, d), ("ca_kv", 2 * d, d),
                                       ("ca_o", d, d), ("up", F, d), ("down", d, F))):
            w[n] = L(1 + 2 * j, o, k)
        return w

    def _angles(self):
        c = self.c
        f, r, k = torch.meshgrid(*(torch.arange(n, device=DEV, dtype=torch.float64)
                                   for n in (c["frames"], c["rows"], c["cols"])), indexing="ij")
        pos = torch.stack([f, r, k], -1).reshape(-1, 3)
        if not self.wan:
            pos = torch.cat([torch.zeros(self.nx, 3, device=DEV, dtype=torch.float64), pos])
        parts = []
        for a, w in enumerate(_axes(c)):
            j = torch.arange(w // 2, device=DEV, dtype=torch.float64)
            parts.append(pos[:, a:a + 1] * 10000.0 ** (-2.0 * j / max(w, 1)))
        return torch.cat(parts, 1)

    def _rope(self, x):
        n = x.shape[0]
        x = x.reshape(n, self.H, self.dh // 2, 2)
        c, s = torch.cos(self.angles)[:, None], torch.sin(self.angles)[:, None]
        return torch.stack([x[..., 0] * c - x[..., 1] * s, x[..., 0] * s + x[..., 1] * c], -1).reshape(n, -1)

    def _rms(self, x, w):
        y = x.reshape(x.shape[0], self.H, self.dh)
        y = y * torch.rsqrt(y.square().mean(-1, keepdim=True) + 1e-6) * w
        return y.reshape(x.shape[0], -1)

    def temb(self, sigma, pooled):
        f = torch.exp(-math.log(10000.0) * torch.arange(TEMB // 2, device=DEV, dtype=torch.float64) / (TEMB // 2))
        a = 1000.0 * sigma * f
        v = _lin(_silu(_lin(torch.cat([torch.cos(a), torch.sin(a)]), self.G["t1"])), self.G["t2"])
        return v if self.wan else v + pooled

    def block_mod(self, b, vec):
        kind, w = self.blocks[b]
        if kind == "single":
            return _lin(_silu(vec), w["mod"])
        if kind == "double":
            return torch.cat([_lin(_silu(vec), w["imgmod"]), _lin(_silu(vec), w["txtmod"])])
        return _lin(_silu(vec), self.G["tproj"]) + w["tab"]

    def apply(self, b, h, vec, ctx=None):
        """Block b on the joint stream (Wan: on the image stream, with its context)."""
        kind, w = self.blocks[b]
        d, nx = self.d, self.nx
        m = self.block_mod(b, vec).reshape(-1, d)
        if kind == "single":
            p = _lin(_lnmod(h, m[0], m[1]), w["lin1"])
            q, k, v = p[:, :d], p[:, d:2 * d], p[:, 2 * d:3 * d]
            if "norm" in w:
                q, k = self._rms(q, w["norm"][0]), self._rms(k, w["norm"][1])
            a = _attend(self._rope(q), self._rope(k), v, self.H)
            return h + m[2] * _lin(torch.cat([a, _gelu(p[:, 3 * d:])], 1), w["lin2"])
        if kind == "double":
            parts = []
            for s, rows, mm in (("txt", h[:nx], m[6:]), ("img", h[nx:], m[:6])):
                p = _lin(_lnmod(rows, mm[0], mm[1]), w[s + "qkv"])
                q, k, v = p[:, :d], p[:, d:2 * d], p[:, 2 * d:]
                if s + "norm" in w:
                    q, k = self._rms(q, w[s + "norm"][0]), self._rms(k, w[s + "norm"][1])
                parts.append((q, k, v))
            q, k, v = (torch.cat(t) for t in zip(*parts))
            a = _attend(self._rope(q), self._rope(k), v, self.H)
            out = []
            for s, rows, aa, mm in (("txt", h[:nx], a[:nx], m[6:]), ("img", h[nx:], a[nx:], m[:6])):
                x = rows + mm[2] * _lin(aa, w[s + "proj"])
                out.append(x + mm[5] * _lin(_gelu(_lin(_lnmod(x, mm[3], mm[4]), w[s + "up"])), w[s + "down"]))
            return torch.cat(out)
        p = _lin(_lnmod(h, m[0], m[1]), w["sa_qkv"])
        a = _attend(self._rope(p[:, :d]), self._rope(p[:, d:2 * d]), p[:, 2 * d:], self.H)
        x = h + m[2] * _lin(a, w["sa_o"])
        kv = _lin(ctx, w["ca_kv"])
        x = x + _lin(_attend(_lin(_lnmod(x), w["ca_q"]), kv[:, :d], kv[:, d:], self.H), w["ca_o"])
        return x + m[5] * _lin(_gelu(_lin(_lnmod(x, m[3], m[4]), w["up"])), w["down"])

    def stack(self, h_img, txt, vec):
        h = h_img if self.wan else torch.cat([txt, h_img])
        for b in range(len(self.blocks)):
            h = self.apply(b, h, vec, txt)
        return h if self.wan else h[self.nx:]

    def final(self, h, vec):
        m = _lin(_silu(vec), self.G["fmod"]).reshape(2, self.d)
        return _lin(_lnmod(h, m[0], m[1]), self.G["fin"])


def _lin(x, wb):
    return x @ wb[0].T + wb[1]


def _silu(x):
    return x * torch.sigmoid(x)


def _gelu(x):
    return 0.5 * x * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (x + 0.044715 * x ** 3)))


def _lnmod(x, shift=None, scale=None):
    y = x - x.mean(-1, keepdim=True)
    y = y * torch.rsqrt(y.square().mean(-1, keepdim=True) + 1e-6)
    return y if shift is None else y * (1.0 + scale) + shift


def _attend(q, k, v, H, rows=4096):
    out = torch.empty_like(q)
    dh = q.shape[1] // H
    for h in range(H):
        c = slice(h * dh, (h + 1) * dh)
        for r in range(0, q.shape[0], rows):
            out[r:r + rows, c] = torch.softmax(q[r:r + rows, c] @ k[:, c].T / math.sqrt(dh), -1) @ v[:, c]
    return out


def _gate_logit(case, layers, x):
    relu = lambda y: np.maximum(y, 0.0)   # noqa: E731
    L = [(w.astype(np.float64), b.astype(np.float64)) for w, b in layers]
    dense = lambda i, y: L[i][0] @ y + L[i][1]   # noqa: E731
    if case["gate_kind"] == "wan6":
        a, b = relu(dense(1, relu(dense(0, x[:3])))), relu(dense(3, relu(dense(2, x[3:]))))
        return float(dense(5, relu(dense(4, np.concatenate([a, b]))))[0])
    for i in range(len(L) - 1):
        x = relu(dense(i, x))
    return float(dense(len(L) - 1, x)[0])


class _UniPC:
    """UniPC of order 2 with its corrector on x = (1 - sigma) x0 + sigma noise, data
    prediction, B(h) = e^-h - 1 (Zhao et al. 2023)."""

    def __init__(self, sig):
        self.sig, self.T = sig, len(sig) - 1
        self.m, self.x, self.used = {}, None, False

    def _lam(self, i):
        return math.log1p(-self.sig[i]) - math.log(self.sig[i])

    def _move(self, i, x, past, new=None):
        """From step i to i + 1; past: the point i - 1 is used; new: m at i + 1 (corrector)."""
        a1, s1, s0 = 1.0 - self.sig[i + 1], self.sig[i + 1], self.sig[i]
        e = s1 * (1.0 - s0) / (a1 * s0)          # e^-h, 0 at either end of the grid
        psi = e - 1.0
        y = s1 / s0 * x - a1 * psi * self.m[i]
        D, r = [], []
        if past:
            r.append((self._lam(i - 1) - self._lam(i)) / -math.log(e) if e > 0 else 0.0)
            if e == 0:
                raise ValueError("the previous point is not used at the ends of the grid")
            D.append((self.m[i - 1] - self.m[i]) / r[0])
        if new is not None:
            r.append(1.0)
            D.append(new - self.m[i])
        if not D:
            return y
        if len(D) == 1:
            rho = [0.5]
        else:
            h = -math.log(e)
            p2 = psi / -h - 1.0
            p3 = p2 / -h - 0.5
            rho = np.linalg.solve(np.array([[1.0, 1.0], r]), np.array([p2 / psi, 2.0 * p3 / psi]))
        return y - a1 * psi * sum(float(c) * t for c, t in zip(rho, D))

    def step(self, i, x, v):
        m = x - self.sig[i] * v
        if i > 0:
            x = self._move(i - 1, self.x, self.used, m)
        self.m[i], self.x = m, x
        self.used = min(2, i + 1, self.T - i) == 2 and self.sig[i - 1] < 1.0
        return self._move(i, x, self.used)


def _exact_sample(case, seed):
    net = _Net(case, seed)
    s = {k: v.double() for k, v in _sample_inputs(case, seed).items()}
    layers, mu, sd = _gate(case, seed)
    T, B, g = case["T"], case["B"], case["guidance"]
    u = [1.0 - i / T for i in range(T + 1)]
    sig = [case["shift"] * w / (1.0 + (case["shift"] - 1.0) * w) for w in u]
    uni = _UniPC(sig) if case["sampler"] == "unipc" else None
    branches = [("txt", "pooled")] + ([("txt_u", "pooled_u")] if g else [])
    x, c, last, R, m_last, m_prev = s["x0"], 0, -1, {}, None, None
    mask, log = np.zeros(T, np.uint8), np.zeros((T, 16))
    for t in range(T):
        vec = {b: net.temb(sig[t], s[b[1]]) for b in branches}
        h_in = _lin(x, net.G["pe"])
        m = h_in
        if case["observable"] == "modulated":
            mod = net.block_mod(0, vec[branches[0]]).reshape(-1, net.d)
            m = _lnmod(h_in, mod[0], mod[1])
        full = 1
        log[t, 4] = 1
        log[t, 6] = c
        if t > 0:
            n1, d1 = float((m - m_last).abs().sum()), float(m_last.abs().sum())
            n2, d2 = float((m - m_prev).abs().sum()), float(m_prev.abs().sum())
            bud = [B / T, (B - c) / B, (B - c) / (T - t)]
            f = [bud[1], (T - t) / T, n1 / d1] if case["gate_kind"] == "mlp3" else bud + [t - last, n1 / d1, n2 / d2]
            z = _gate_logit(case, layers, (np.array(f) - mu) / sd)
            full = bit = int(z > 0)
            full = 1 if B - c >= T - t else full
            full = 0 if B == c else full
            log[t] = [bud[1], (T - t) / T, n1 / d1, z, bit, full, c, t - last, *bud, n1, d1, n2 / d2, n2, d2]
        log[t, 5] = mask[t] = full
        vel = []
        for b in branches:
            if full:
                R[b] = net.stack(h_in, s[b[0]], vec[b]) - h_in
            vel.append(net.final(h_in + R[b], vec[b]))
        if full:
            c, last, m_last = c + 1, t, m
        m_prev = m
        v = vel[1] + g * (vel[0] - vel[1]) if g else vel[0]
        x = uni.step(t, x, v) if uni else x + (sig[t + 1] - sig[t]) * v
    return x, mask, log


def exact(case, seed):
    op = case["op"]
    # float64 products of 1 to 2 TFLOP/s: keep a case within some ten seconds
    if op in MODEL_OPS and work(case)["flops"] > 1.5e13 or op == "attention" and work(case)["flops"] > 1e13:
        return None
    if op in ("sample", "steps"):
        x, mask, log = _exact_sample(case, seed)
        return {"latent": x, "mask": mask, "log": log} if op == "sample" else {"latent": x, "flags": mask.astype(np.int32)}
    if op == "block":
        net, s = _Net(case, seed), _sample_inputs(case, seed)
        u = 1.0 - (case["T"] // 2) / case["T"]
        sigma = case["shift"] * u / (1.0 + (case["shift"] - 1.0) * u)
        return net.apply(0, _block_input(case, seed).double(), net.temb(sigma, s["pooled"].double()), s["txt"].double())
    s = _op_inputs(case, seed)
    if op == "attention":
        v = s["vt"][:, :, :case["nk"]].double().permute(2, 0, 1).reshape(case["nk"], -1)
        return _attend(s["q"].double(), s["k"].double(), v, case["heads"])
    if op == "mlp":
        return torch.cat([_gelu(a.double() @ s["W"].double().T + s["bias"].double()) for a in s["A"].split(512)])
    if op == "norm":
        return _lnmod(s["x"].double(), s["shift"].double(), s["scale"].double())
    a, b = s["a"].double(), s["b"].double()
    num, den = (a - b).abs().sum(), b.abs().sum()
    return torch.stack([num / den, num, den])
