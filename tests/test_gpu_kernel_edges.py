"""GPU kernels at the sizes where they can go wrong (tile edges, remainders, the smallest
and largest of a range), against the fp64 oracle or a plain fp64 restatement of the op."""

import ctypes

import numpy as np
import pytest
import torch

from oracle import bag_oracle as O
from paper_2608_09231_gb300 import bag, configs, synth

pytestmark = pytest.mark.gpu


def call_us(call, n):
    """Microseconds a call, the least of eight loops of n calls."""
    best = 1e9
    for _ in range(8):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(n):
            call()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * e0.elapsed_time(e1) / n)
    return best


@pytest.mark.parametrize("gate_kind", ["mlp3", "flux6", "wan6"])
@pytest.mark.parametrize("grid", [(1, 1, 1), (1, 1, 127), (1, 8, 16), (1, 3, 43), (1, 33, 31), (1, 32, 32), (1, 25, 61)])
def test_gate_reduction_and_logit_at_thread_edges(grid, gate_kind, lib):
    """Row counts around the gate's 128 and, from 1024 rows, 512 threads (1, 127, 128, 129, 1023,
    1024, 1525): the logged drift and step change against the oracle's (fp32 sums of fp32 row sums: relative error under
    1e-5), the logit bit for bit on the logged inputs, the decisions from the logged bits."""
    cfg = configs.get_config("tiny", grid=grid, n_txt=5, gate_kind=gate_kind, n_single=1)
    T, B = 4, 2
    ctx = bag.create(cfg, T=T, B=B)
    inp = synth.make_inputs(cfg)
    x = torch.from_numpy(inp["x"].copy()).cuda()
    m, log, nfe = ctx.run(x, torch.from_numpy(inp["txt"]).cuda(), torch.from_numpy(inp["pooled"]).cuda())
    ctx.close()
    g = synth.make_gate_any(cfg["gate_seed"], gate_kind)
    ref = O.sample(cfg, synth.make_weights(cfg), g, inp, T=T, B=B, policy=[int(v) for v in m])
    assert nfe == B and list(m) == O.schedule_from_gate_bits([None] + [int(v) for v in log[1:, 4]], B, T)
    for t in range(1, T):
        drift, step = ref["log"][t]["drift"], ref["log"][t]["s_traj"][2]
        assert abs(float(log[t, 2]) - drift) <= 1e-5 * drift and abs(float(log[t, 13]) - step) <= 1e-5 * step
        cols = [0, 1, 2] if gate_kind == "mlp3" else [8, 9, 10, 7, 2, 13]
        f = [np.float32(v) for v in log[t, cols]]
        z = O.gate_logit(f, g) if gate_kind == "mlp3" else O.gate_logit6(f, g)
        assert z == np.float32(log[t, 3]) and bool(log[t, 4]) == bool(z > 0), t


@pytest.mark.parametrize("heads,hidden,grid,n_txt", [
    (2, 128, (1, 1, 1), 1),      # 2 tokens: one query group, one key tile, seven warps without keys
    (2, 128, (1, 3, 9), 5),      # 32 tokens: whole tiles
    (3, 192, (1, 4, 7), 5),      # 33 tokens: one row and one key past a tile
    (2, 256, (1, 1, 250), 7),    # 257 tokens, head width 128: a second round of key tiles
    (2, 128, (1, 1, 249), 7),    # 256 and 257 tokens: eight warps, twelve
    (2, 128, (1, 1, 250), 7),
    (2, 128, (1, 1, 377), 7),    # 384 and 385 tokens: the last with twelve, a second round of the eight
    (2, 128, (1, 1, 378), 7),
    (4, 256, (1, 1, 297), 7),    # 304 and 305 tokens x 4 heads: a CTA per SM, one more row of CTAs
    (4, 256, (1, 1, 298), 7),
    (2, 128, (1, 17, 29), 20),   # 513 tokens
])
def test_fp32_backbone_at_tile_edges(heads, hidden, grid, n_txt, lib):
    """The fp32 projections (32 x 32 tiles, K in slices of 64 split over eight warps) and the
    fp32 attention (eight queries a CTA, key tiles of 32 over eight or twelve warps): latents against
    the fp64 oracle to 1e-5 of their RMS (fp32 sums over up to 640 products)."""
    dh = hidden // heads
    cfg = configs.get_config("tiny", hidden=hidden, heads=heads, mlp=4 * hidden, grid=grid, n_txt=n_txt, n_single=1,
                             rope_axes=(0, 32, 32) if dh == 64 else (16, 56, 56))
    ctx = bag.create(cfg, T=2, B=2)
    inp = synth.make_inputs(cfg)
    x = torch.from_numpy(inp["x"].copy()).cuda()
    ctx.run(x, torch.from_numpy(inp["txt"]).cuda(), torch.from_numpy(inp["pooled"]).cuda())
    ctx.close()
    ref = O.sample(cfg, synth.make_weights(cfg), synth.make_gate(cfg["gate_seed"]), inp, T=2, B=2)["x"]
    rms = float(np.sqrt(np.mean(ref ** 2)))
    assert float(np.max(np.abs(x.cpu().numpy() - ref))) <= 1e-5 * rms


@pytest.mark.parametrize("M,N,K", [(1, 64, 64), (33, 64, 192), (31, 128, 320), (65, 192, 1024)])
@pytest.mark.parametrize("offset", [0, 1, 4])  # 16-byte rows and not
def test_cuda_core_gemm_of_bf16_rows(M, N, K, offset, lib):
    """One K slice, a ring's worth and more, with 16-byte loads and single ones, against fp64:
    the fp32 sum over K, bounded by 4 K 2^-24 sum|a||w|; rows around the operands hold NaN."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(M + N + K + offset)

    def rows(n):
        buf = torch.full((n + 2, K + offset), float("nan"), device="cuda").bfloat16()
        buf[1:n + 1, offset:] = torch.randn(n, K, generator=g, device="cuda").bfloat16()
        return buf[1:n + 1, offset:]

    A, W, C = rows(M), rows(N), torch.full((M + 1, N), -7.0, device="cuda")
    ctx.gemm_bf16(A, W, None, C, M, N, K, 0, 1)
    torch.cuda.synchronize()
    ctx.close()
    err = (C[:M].double() - A.double() @ W.double().T).abs()
    assert bool((err <= 4 * K * 2.0 ** -24 * (A.double().abs() @ W.double().abs().T)).all())
    assert bool((C[M] == -7.0).all())


def test_cuda_core_gemm_of_bf16_rows_keeps_its_time(lib):
    """2048 x 2048 x 2048: no more than the 753 us of 64 x 64 tiles (507 with operands fetched a
    slice ahead, 988 without)."""
    ctx = bag.create("tiny", T=2, B=1)
    A, W = (torch.randn(2048, 2048, device="cuda").bfloat16() for _ in range(2))
    C = torch.empty(2048, 2048, device="cuda")
    us = call_us(lambda: ctx.gemm_bf16(A, W, None, C, 2048, 2048, 2048, 0, 1), 10)
    ctx.close()
    assert us <= 753, us


@pytest.mark.parametrize("n,nk,heads,dh", [(9, 30, 2, 64), (33, 70, 1, 128), (40, 300, 2, 64)])
@pytest.mark.parametrize("transposed", [0, 1])
@pytest.mark.parametrize("offset", [0, 1, 4])  # 8-byte rows and not
def test_cuda_core_attention_of_bf16_rows(n, nk, heads, dh, transposed, offset, lib):
    """Vector loads and single ones, against fp64 (fp32 throughout, the output's bf16 rounding);
    what lies past the last key of a transposed V holds NaN."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(n + nk + offset)
    ld = heads * dh + offset

    def rows(m):
        return torch.randn(m * ld + offset, generator=g, device="cuda").bfloat16()[offset:].view(m, ld)

    q, k, v = rows(n), rows(nk), rows(nk)
    vpad = (nk + 8) // 8 * 8 if transposed else 0
    vv = v
    if transposed:
        vv = torch.full((heads * dh * vpad + offset,), float("nan"), device="cuda").bfloat16()[offset:].view(-1, vpad)
        vv[:, :nk] = v[:, :heads * dh].T
    o = torch.full((n + 1, ld), 9.0, device="cuda").bfloat16()
    ctx.attention_bf16(q, k, vv, o, n, nk, heads, dh, vpad, 1)
    torch.cuda.synchronize()
    ctx.close()
    for h in range(heads):
        c = slice(h * dh, h * dh + dh)
        ref = torch.softmax(q[:, c].double() @ k[:, c].double().T / dh ** 0.5, -1) @ v[:, c].double()
        assert bool(((o[:n, c].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5).all()), h
    assert bool((o[n] == 9.0).all()) and bool((o[:, heads * dh:] == 9.0).all())


@pytest.mark.parametrize("cols", [4, 508, 3072, 3076, 5116, 5120, 5124, 6144])
def test_ln_mod_widths(cols, lib):
    """Around each change of threads and columns a thread (128 threads to 3072 columns, 256 with
    five or six float4 each past it), the narrowest and the widest row: the output's bf16 rounding
    and fp32 statistics; the rows around it stay untouched."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(cols)
    x = 2.0 * torch.randn(5, cols, generator=g, device="cuda") + 0.5
    sh, sc = (0.5 * torch.randn(cols, generator=g, device="cuda") for _ in range(2))
    y = torch.full((7, cols), 9.0, device="cuda").bfloat16()
    ctx.ln_mod(x, sh, sc, y[1:], 5, cols)
    torch.cuda.synchronize()
    ctx.close()
    xd = x.double()
    ref = (xd - xd.mean(1, keepdim=True)) / (xd.var(1, unbiased=False, keepdim=True) + 1e-6).sqrt()
    ref = ref * (1 + sc.double()) + sh.double()
    assert bool(((y[1:6].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5).all())
    assert bool((y[0] == 9.0).all() and (y[6] == 9.0).all())


def test_signal_and_cache_passes_of_wide_rows(lib):
    """The signal pass and the final layer's pass with the residual cache past 5120 columns (six
    float4 a thread): a sample with reused steps at width 5248 against the fp64 oracle, to the
    2e-2 x RMS of bf16 operands, and the logged drift to 1e-2 (bf16 observables)."""
    cfg = configs.get_config("tiny", hidden=5248, heads=41, mlp=1024, dtype="bf16", grid=(1, 3, 7), n_txt=5,
                             n_single=1, rope_axes=(16, 56, 56))
    mask = [1, 0, 0, 1, 0]
    inp = synth.make_inputs(cfg)
    ctx = bag.create(cfg, T=5, B=2)
    ctx.set_policy(bag.POLICY_MASK, np.array(mask, np.uint8))
    x = torch.from_numpy(inp["x"].copy()).cuda()
    m, log, nfe = ctx.run(x, torch.from_numpy(inp["txt"]).cuda().bfloat16(), torch.from_numpy(inp["pooled"]).cuda())
    ctx.close()
    assert list(m) == mask and nfe == 2
    inp["txt"] = synth.bf16_round(inp["txt"])
    ref = O.sample(cfg, synth.make_weights(cfg), synth.make_gate(cfg["gate_seed"]), inp, T=5, B=2, policy=mask)
    rms = float(np.sqrt(np.mean(ref["x"] ** 2)))
    assert float(np.max(np.abs(x.cpu().numpy() - ref["x"]))) <= 2e-2 * rms
    for t in range(1, 5):
        assert abs(float(log[t, 2]) - ref["log"][t]["drift"]) <= 1e-2 * ref["log"][t]["drift"], t


def test_cuda_core_attention_of_bf16_rows_keeps_its_time(lib):
    """1024 tokens x 8 heads of 64: no more than the 203 us of the kernel that staged keys and
    values in shared memory (145 with vector loads, 330 with single ones)."""
    ctx = bag.create("tiny", T=2, B=1)
    q, k, v = (torch.randn(1024, 512, device="cuda").bfloat16() for _ in range(3))
    o = torch.empty_like(q)
    us = call_us(lambda: ctx.attention_bf16(q, k, v, o, 1024, 1024, 8, 64, 0, 1), 20)
    ctx.close()
    assert us <= 203, us


@pytest.mark.parametrize("nk", [1, 33, 34, 36, 289])  # one to three keys past a group of four, none
@pytest.mark.parametrize("transposed", [0, 1])
@pytest.mark.parametrize("dh", [64, 128])
def test_cuda_core_attention_with_an_infinite_value(nk, transposed, dh, lib):
    """An infinity in the last key's value makes that column infinite (every weight is positive
    here), not NaN, and no other."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(nk)
    q, k, v = (torch.randn(n, dh, generator=g, device="cuda").bfloat16() for n in (9, nk, nk))
    v[nk - 1, 3] = float("inf")
    vpad = (nk + 7) // 8 * 8 if transposed else 0
    vv = v
    if transposed:
        vv = torch.zeros(dh, vpad, device="cuda", dtype=torch.bfloat16)
        vv[:, :nk] = v.T
    o = torch.zeros(9, dh, device="cuda", dtype=torch.bfloat16)
    ctx.attention_bf16(q, k, vv, o, 9, nk, 1, dh, vpad, 1)
    torch.cuda.synchronize()
    ctx.close()
    want = torch.softmax(q.double() @ k.double().T / dh ** 0.5, -1) @ v.double()
    assert bool(torch.isinf(o[:, 3]).all()) and bool(torch.isfinite(want[:, 4:]).all())
    rest = [c for c in range(dh) if c != 3]
    err = (o.double() - want)[:, rest].abs()
    # fp32 throughout, the output's bf16 rounding
    assert bool((err <= 2.0 ** -8 * want[:, rest].abs() + 1e-5).all())


def test_attention_of_few_rows_takes_the_short_way_out(lib):
    """Device time (captured) of 64 queries x 64 keys: two heads against 48, whose output goes
    through shared memory as the two heads' once did (0.98 of the time then, 0.86 now)."""
    ctx = bag.create("tiny", T=2, B=1)
    s = torch.cuda.Stream()
    ctx.set_stream(s.cuda_stream)
    graphs, keep = [], []
    for heads in (2, 48):
        q, k = (torch.randn(64, heads * 128, device="cuda").half() for _ in range(2))
        vt, o = torch.randn(heads, 128, 128, device="cuda").half(), torch.empty(64, heads * 128, device="cuda").bfloat16()
        keep.append((q, k, vt, o))
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1], stream=s):
            for _ in range(40):
                ctx.attention_f16(q, k, vt, o, 64, 64, heads, 128, 128)
    us = [1e9, 1e9]
    for _ in range(30):  # in turn: the clock is the same for both
        for i, graph in enumerate(graphs):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(5):
                graph.replay()
            e1.record()
            torch.cuda.synchronize()
            us[i] = min(us[i], e0.elapsed_time(e1) * 5)
    del graphs
    ctx.close()
    assert us[0] <= 0.92 * us[1], us


def test_fp32_attention_of_twice_the_tokens(lib):
    """From 256 to 512 tokens x 4 heads (four times the work, launches that fill the GPU once and
    twice): 1.9 times the time with eight warps a CTA, 2.6 with twelve at the larger one."""
    us = []
    for n in (256, 512):
        cfg = configs.get_config("tiny", grid=(1, 1, n - 16), n_txt=16, n_single=1)
        ctx = bag.create(cfg, T=8, B=8)
        inp = synth.make_inputs(cfg)
        txt, pooled = torch.from_numpy(inp["txt"]).cuda(), torch.from_numpy(inp["pooled"]).cuda()
        best = 1e9
        for _ in range(6):
            ctx.reset()
            ctx.profile_run(torch.from_numpy(inp["x"].copy()).cuda(), txt, pooled)
            best = min([best] + [r["ms"] for r in ctx.profile_launches() if r["kind"] == "attention"])
        ctx.close()
        us.append(1e3 * best)
    assert us[1] <= 2.25 * us[0], us


@pytest.mark.parametrize("M,N,K", [
    (1, 64, 64 * 7),      # seven K blocks: not split
    (1, 64, 512),         # the least that is: one row, four CTAs of two K blocks
    (127, 64, 64 * 9),    # four CTAs, one with three blocks
    (129, 128, 64 * 17),  # four CTAs, four or five blocks each, one row in the last row tile
    (300, 192, 64 * 35),  # nine tiles, eight or nine blocks each
    (2432, 128, 512),     # 38 tiles, the most for four CTAs
    (1650, 192, 512),     # 39 tiles: two CTAs of four blocks
    (1100, 512, 64 * 17), # 72 tiles, two CTAs, eight and nine blocks
    (1100, 512, 1024),    # even shares
    (2400, 256, 64 * 9),  # 76 tiles, the most for two CTAs, four and five blocks
    (1400, 448, 64 * 9),  # 77 tiles: not split
    (640, 1024, 2048),    # 80 tiles: not split
])
@pytest.mark.parametrize("epilogue", [0, 1])
def test_split_k_gemm(M, N, K, epilogue, lib):
    """Shapes around the split-K rule (tiles x CTAs against 152 SMs, at least eight K blocks)
    against fp64: a bf16 product's fp32 sum over K, bounded by 4 K 2^-24 sum|a||w|."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    W = (0.05 * torch.randn(N, K, generator=g, device="cuda")).bfloat16()
    bias = 0.1 * torch.randn(N, generator=g, device="cuda")
    C = torch.full((M + 1, N), -7.0, device="cuda")
    ctx.gemm_bf16(A, W, bias, C, M, N, K, epilogue)
    torch.cuda.synchronize()
    ctx.close()
    ref = A.double() @ W.double().T + bias.double()
    # GELU's slope is at most 1.13
    bound = 1.2 * (4 * K * 2.0 ** -24 * (A.double().abs() @ W.double().abs().T) + 1e-6)
    if epilogue:
        ref = torch.nn.functional.gelu(ref, approximate="tanh")
    assert bool(((C[:M].double() - ref).abs() <= bound).all())
    assert bool((C[M] == -7.0).all())


@pytest.mark.parametrize("M,N", [(32, 1024), (32, 4096)])
def test_gemm_of_four_k_blocks_costs_no_more_than_three(M, N, lib):
    """Around the K block count where a launch starts to split K: the call with one block more
    (split in two it took 1.3 to 1.4 times as long)."""
    ctx = bag.create("tiny", T=2, B=1)
    us = []
    for K in (192, 256):
        A, W = torch.randn(M, K, device="cuda").bfloat16(), torch.randn(N, K, device="cuda").bfloat16()
        C = torch.empty(M, N, device="cuda")
        us.append(call_us(lambda: ctx.gemm_bf16(A, W, None, C, M, N, K), 100))
    ctx.close()
    assert us[1] <= 1.2 * us[0], us


@pytest.mark.parametrize("M,N,K", [
    (33, 64, 128), (1300, 1280, 64),     # 128 x 64 tiles: one, 110 x 2 of them
    (33, 64, 512), (1100, 512, 576),     # K split over four CTAs, over two
    (1300, 1920, 64), (1217, 2176, 448), # 128 x 128 tiles: 165, and 170 with one row in the last row tile
    (2500, 3072, 64),                    # CTA pairs, eight epilogue warps
    (2500, 3072, 1088),                  # four (17 K blocks)
])
@pytest.mark.parametrize("epilogue", [0, 1])
@pytest.mark.parametrize("offset,pad", [(0, 0), (4, 4), (1, 3)])  # 16-byte rows and not
def test_fp32_output_rows(M, N, K, epilogue, offset, pad, lib):
    """fp32 outputs through the transposing epilogue and, for rows that are not 16-byte
    aligned, through the per-row one; columns and rows around the output stay untouched."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    W = (0.1 * torch.randn(N, K, generator=g, device="cuda")).bfloat16()
    bias = 0.1 * torch.randn(N, generator=g, device="cuda")
    whole = torch.full((M + 1, N + offset + pad), -7.0, device="cuda")
    ctx.gemm_bf16(A, W, bias, whole[:M, offset:offset + N], M, N, K, epilogue)
    torch.cuda.synchronize()
    ctx.close()
    ref = A.double() @ W.double().T + bias.double()
    bound = 1.2 * (4 * K * 2.0 ** -24 * (A.double().abs() @ W.double().abs().T) + 1e-6)
    if epilogue:
        ref = torch.nn.functional.gelu(ref, approximate="tanh")
    assert bool(((whole[:M, offset:offset + N].double() - ref).abs() <= bound).all())
    assert bool((whole[M] == -7.0).all() and (whole[:, :offset] == -7.0).all() and (whole[:, offset + N:] == -7.0).all())


@pytest.mark.parametrize("rows,cols", [
    (1, 1), (3, 8), (129, 256),   # one cluster: fewer rows than warps
    (256, 127), (256, 256),       # a row a warp; elements, 16-byte groups, the byte limit (fp32)
    (256, 129), (257, 64), (128, 513), (256, 264),  # just past a limit: elements, rows, width (fp32), bytes (fp32)
    (300, 255),                   # rows that are not 16-byte groups
    (1, 65536), (8, 16384),       # few bytes in wide rows: four warps a row
    (1215, 520), (1217, 1023),    # around a warp per row (eight rows an SM)
    (64, 40000), (4099, 130)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("offset", [0, 1])  # inputs and scratch off 16-byte alignment
def test_rel_l1_routes(rows, cols, dtype, offset, lib):
    """Every route of the relative L1 (cluster, four warps or one a row; 16-byte groups or
    elements): sums against fp64 to 2e-6 (fp32 chains of at most 512 terms, each rounding at
    most 2^-24 of the sum and of either sign, then a tree), the same bits again and through the
    allocation-free entry."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(rows * 7 + cols)

    def tensor():
        buf = torch.randn(rows * cols + offset, generator=g, device="cuda").to(dtype)
        return buf[offset:].reshape(rows, cols)

    a, b = tensor(), tensor()
    scratch = torch.zeros(2 * rows + 2, device="cuda")
    out, again, noalloc = (torch.zeros(3, device="cuda") for _ in range(3))
    ctx.rel_l1(a, b, rows, cols, scratch[offset:], out)
    ctx.rel_l1(a, b, rows, cols, scratch[offset:], again)
    torch.cuda.synchronize()
    bag.rel_l1_noalloc(a, b, rows, cols, noalloc)
    torch.cuda.synchronize()
    ctx.close()
    num, den = (a.double() - b.double()).abs(), b.double().abs()
    ref = torch.stack([num.sum() / den.sum(), num.sum(), den.sum()])
    assert bool(((out.double() - ref).abs() <= 2e-6 * ref).all())
    part = scratch[offset:offset + 2 * rows].reshape(rows, 2).double()
    assert bool(((part[:, 0] - num.sum(1)).abs() <= 2e-6 * num.sum(1)).all())
    assert bool(((part[:, 1] - den.sum(1)).abs() <= 2e-6 * den.sum(1)).all())
    assert float(scratch[offset + 2 * rows]) == 0.0
    assert torch.equal(out, again) and torch.equal(out, noalloc)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_rel_l1_is_as_exact_in_one_launch(dtype, lib):
    """Relative error of the three sums over 80 inputs of 256 x 256 (root mean square): at most
    52e-9, where two launches have 41e-9 to 47e-9 (a chain over the eight CTAs' sums had 55e-9 to
    60e-9, a tree has 45e-9 to 48e-9; 240 values, so each is known to about 5 %)."""
    out, err = torch.zeros(3, device="cuda"), []
    for seed in range(80):
        g = torch.Generator(device="cuda").manual_seed(seed)
        b = torch.randn(256, 256, generator=g, device="cuda")
        a = (b + 0.2 * torch.randn(256, 256, generator=g, device="cuda")).to(dtype)
        b = b.to(dtype)
        bag.rel_l1_noalloc(a, b, 256, 256, out)
        torch.cuda.synchronize()
        num, den = (a.double() - b.double()).abs().sum(), b.double().abs().sum()
        err.append(out.double() / torch.stack([num / den, num, den]) - 1)
    assert float(torch.stack(err).square().mean().sqrt()) <= 52e-9


@pytest.mark.parametrize("rows,cols", [(64, 64), (300, 64), (1300, 64)])  # one launch, two (four warps a row, one)
def test_a_failed_launch_leaves_no_error_to_the_next_call(rows, cols, lib):
    """A launch on a stream whose capture was invalidated fails on the host; the next call, on
    another stream, succeeds.  (Synchronising a stream that is being captured invalidates it.)"""
    ctx = bag.create("tiny", T=2, B=1)
    a, out = torch.randn(rows, cols, device="cuda"), torch.zeros(3, device="cuda")
    total, n = torch.zeros_like(a), rows * cols
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    driver, handle, graph = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
    bag.rel_l1_noalloc(a, a, rows, cols, out)  # looks up its scratch outside the capture
    torch.cuda.synchronize()
    assert driver.cuStreamBeginCapture_v2(handle, 2) == 0  # relaxed: no other stream or thread is concerned
    assert driver.cuStreamSynchronize(handle) != 0
    with pytest.raises(bag.BagError):
        bag.rel_l1_noalloc(a, a, rows, cols, out, s.cuda_stream)
    assert driver.cuStreamEndCapture(handle, ctypes.byref(graph)) != 0
    ctx.residual_add(total, a, a, n)
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(total, a + a)


@pytest.mark.parametrize("dtype,cols", [(torch.float32, 65536), (torch.bfloat16, 131072)])
@pytest.mark.parametrize("offset", [0, 1])
def test_rel_l1_of_one_wide_row_is_not_left_to_one_warp(dtype, cols, offset, lib):
    """512 KB in one row take less time than the 1 MB of a row twice as wide, whose route does
    not depend on the size (one warp alone took 49 to 320 us for the former, against 46 to 52)."""
    us = []
    for n in (cols, 2 * cols):
        a, b = (torch.randn(n + offset, device="cuda").to(dtype)[offset:].reshape(1, n) for _ in range(2))
        out = torch.zeros(3, device="cuda")
        us.append(call_us(lambda: bag.rel_l1_noalloc(a, b, 1, n, out), 50))
    assert us[0] <= 0.8 * us[1], us


@pytest.mark.parametrize("nq,nk,heads", [
    (100, 1408, 1),    # 11 key tiles: not shared
    (100, 1536, 2),    # four CTAs a unit, three tiles each
    (257, 1537, 3),    # one key in the 13th tile, one row in the last query pair
    (10240, 2049, 1),  # 40 units: two CTAs, eight or nine tiles
    (2560, 2000, 16),  # 160 units on 152 SMs: the last eight are shared
    (1, 1, 1),         # one row, one key
    (128, 130, 20),    # the most rows written a row a lane
    (128, 64, 21),     # and past it: through shared memory
    (129, 128, 2),     # one row in the second tile of the pair
])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_attention_shared_units_and_few_rows(nq, nk, heads, dtype, lib):
    """Units shared by a cluster, and few rows, against fp64: the output's bf16 rounding (2^-8
    relative) plus the operand type's rounding of P (2^-11 or 2^-8 of the largest output)."""
    ctx = bag.create("tiny", T=2, B=1)
    g = torch.Generator(device="cuda").manual_seed(nq + nk)
    q, k, v = (torch.randn(n, heads, 128, generator=g, device="cuda").to(dtype) for n in (nq, nk, nk))
    vpad = (nk + 127) // 128 * 128
    vt = torch.zeros(heads, 128, vpad, device="cuda", dtype=dtype)
    vt[:, :, :nk] = v.permute(1, 2, 0)
    o = torch.full((nq + 1, heads * 128), 9.0, device="cuda", dtype=torch.bfloat16)
    call = ctx.attention_f16 if dtype == torch.float16 else ctx.attention_bf16
    call(q.reshape(nq, -1), k.reshape(nk, -1), vt, o, nq, nk, heads, 128, vpad)
    torch.cuda.synchronize()
    ctx.close()
    for h in range(heads):
        p = torch.softmax(q[:, h].double() @ k[:, h].double().T / 128 ** 0.5, -1)
        ref = p @ v[:, h].double()
        err = (o[:nq, 128 * h:128 * h + 128].double() - ref).abs()
        share = 2.0 ** -10 if dtype == torch.float16 else 2.0 ** -8
        assert bool((err <= 2.0 ** -8 * ref.abs() + share * ref.abs().max()).all()), h
    assert bool((o[nq] == 9.0).all())
