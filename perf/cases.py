"""The work that a serving program has this library do, as cases that can be timed and compared.

Five kinds of call, each through the public entry points of `paper_2503_24358_b200`:

  prefill   one layer's prompt: the subspace from the prompt's queries (SVD or block power method), then keys and
            values of the whole batch quantized into the cache.  Once per layer and prompt.
  window    one decode window: the residual buffer's keys and values quantized into the cache at their offset, with the
            update matrices of the prompt.  Once per layer and R generated tokens.
  attend    one decode step of attention over the packed cache and the residual buffer.  Once per layer and token.
  readback  keys and values of a cache dequantized, as for a recomputation or a move to another engine.
  host      the prefill of a layer whose tensors are in host memory (offloaded), copies included.

Sizes: the library's own five workloads (squat_inputs/configs.py) and others of the same ranges, with token counts that
are not powers of two.  Head dimension 128 throughout (the only one built).
"""
import math

import torch

import paper_2503_24358_b200 as sq
from squat_inputs.configs import CONFIGS

D = 128
LAMBDA = CONFIGS[1].lam

# Head layouts (query heads, KV heads) of the workloads: tiny, multi-head, grouped-query.
HEADS = ((8, 8), (32, 32), (32, 8))

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
METAS = {"f32": torch.float32, "f16": torch.float16}


def _case(kind, batch, q_heads, kv_heads, tokens, bits=2, group=32, meta="f32", dtype="bf16", **more):
    return dict(kind=kind, batch=batch, q_heads=q_heads, kv_heads=kv_heads, tokens=tokens, bits=bits, group=group,
                meta=meta, dtype=dtype, **more)


def _named(name, c):
    return dict(c, name=name)


def listed():
    return [
        # The smallest prompt: workload 0 as it stands (8 heads, 256 tokens, float32, rank 8), where launches and the
        # latency of the small factorisations are all there is.
        _named("prefill-tiny-f32", _case("prefill", 1, 8, 8, 256, dtype="f32", rank=8, block=1, step1="svd")),
        # Workload 1: one Llama-2-7B-shaped layer, a 4096-token prompt, the paper's default options.
        _named("prefill-7b-4096", _case("prefill", 1, 32, 32, 4096, rank=32, block=1, step1="svd")),
        # Workload 2's layer (grouped-query, batch 16) at a ragged length, with the settings of the paper's experiments:
        # block updates of 64 channels, 16-bit scales; step 1 by the block power method, the fast option.
        _named("prefill-gqa-power", _case("prefill", 16, 32, 8, 8160, meta="f16", rank=32, block=64, step1="power")),
        # Workload 4: long context, the sweep's corner with 4 bits, rank 64 and groups of 128.
        _named("prefill-long-4bit", _case("prefill", 4, 32, 32, 32768, bits=4, group=128, rank=64, block=1, step1="svd")),
        # A decode window of a single sequence: 4096 key vectors into the cache of one layer.
        _named("window-single", _case("window", 1, 32, 32, 128, rank=32, block=1, cache=2048)),
        # Workload 3: the decode window of 64 sequences, into their 4096-token caches.
        _named("window-batch64", _case("window", 64, 32, 32, 128, rank=32, block=1, cache=4096)),
        # Decode step of a single sequence after workload 1's prompt, residual buffer full.
        _named("attend-single", _case("attend", 1, 32, 32, 4096, residual=128, rope=False)),
        # Decode step of workload 2's batch: four query heads share a KV head; 16-bit scales, odd residual length.
        _named("attend-gqa-b16", _case("attend", 16, 32, 8, 8160, meta="f16", residual=57, rope=False)),
        # Decode step of workload 3's batch over full 4096-token caches.
        _named("attend-batch64", _case("attend", 64, 32, 32, 4096, residual=128, rope=False)),
        # Decode step over keys stored before the rotary embedding, 4 bits, groups of 64, a few sequences.
        _named("attend-rope-4bit", _case("attend", 5, 32, 32, 3520, bits=4, group=64, residual=45, rope=True)),
        # The cache of workload 1 read back to bf16.
        _named("readback-7b-4096", _case("readback", 1, 32, 32, 4096)),
        # Workload 1 from pinned host buffers, results back to the host.
        _named("host-prefill-7b", _case("host", 1, 32, 32, 4096, rank=32, block=1, step1="svd")),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind, a head layout, options as the sweep of workload 4 and the paper's experiments vary them,
    and a batch and a token count spread over the logarithm of their ranges."""
    kind = rng.choice(("prefill", "prefill", "prefill", "window", "window", "attend", "attend", "attend", "readback", "host"))
    qh, kvh = rng.choice(HEADS)
    bits, group = rng.choice((2, 2, 4)), rng.choice((32, 32, 64, 128))
    meta, dtype = rng.choice(("f32", "f16")), rng.choice(("bf16", "bf16", "f32"))
    more = {}
    if kind in ("prefill", "host"):
        more = dict(rank=rng.choice((8, 32, 32, 64)), block=rng.choice((1, 1, 32, 64)), step1=rng.choice(("svd", "svd", "power")))
        batch = _log_int(rng, 1, 16) if kind == "prefill" else 1
        most = (1 << 22 if dtype == "bf16" else 1 << 21) if kind == "prefill" else (1 << 17 if dtype == "bf16" else 1 << 16)
        tokens = _log_int(rng, 256, min(32768, most // (batch * kvh)))
    elif kind == "window":
        more = dict(rank=rng.choice((8, 32, 32, 64)), block=rng.choice((1, 1, 32, 64)))
        batch, tokens = _log_int(rng, 1, 64 if dtype == "bf16" else 32), rng.choice((1, 2, 4)) * max(group, 32)
        tokens = min(tokens, 128)
        more["cache"] = tokens * rng.randint(2, 16)
    elif kind == "attend":
        batch = _log_int(rng, 1, 64)
        tokens = _log_int(rng, 128, min(32768, (1 << 23) // (batch * kvh * (bits // 2))))
        more = dict(residual=rng.randint(0, 128), rope=rng.random() < 0.25)
    else:
        batch = _log_int(rng, 1, 16)
        tokens = _log_int(rng, 256, min(32768, (1 << 21) // (batch * kvh)))
    return _case(kind, batch, qh, kvh, max(1, tokens // group) * group, bits, group, meta, dtype, **more)


# ------------------------------------------------------------------------------------------------------------ inputs
def _queries(c, g):
    """Prompt queries of one sample, A B + 0.1 N: a low-rank part that the heads of a KV group share, and noise."""
    rho = 24 if c["q_heads"] != c["kv_heads"] else 16
    qh, kvh, n = c["q_heads"], c["kv_heads"], c["prompt"] if "prompt" in c else c["tokens"]
    basis = torch.randn((kvh, 1, rho, D), generator=g, device="cuda")
    a = torch.randn((kvh, qh // kvh, n, rho), generator=g, device="cuda")
    q = torch.matmul(a.double(), basis.double()).float().view(qh, n, D)
    q += 0.1 * torch.randn((qh, n, D), generator=g, device="cuda")
    return q.to(DTYPES[c["dtype"]])


def _normal(shape, g, dtype, outliers=None):
    """Standard normal rows, sample by sample; `outliers` [heads, d] scales the outlier channels of keys."""
    x = torch.empty(shape, dtype=dtype, device="cuda")
    for b in range(shape[0]):
        y = torch.randn(shape[1:], generator=g, device="cuda")
        if outliers is not None:
            y *= outliers[:, None, :]
        x[b] = y
    return x


def _outliers(kvh, g):
    m = torch.ones((kvh, D), device="cuda")
    at = torch.rand((kvh, D), generator=g, device="cuda").argsort(1)[:, :4]
    return m.scatter_(1, at, 10.0)


def _key_cache(c, tokens, device="cuda", pin=False):
    B, H, G = c["batch"], c["kv_heads"], c["group"]
    new = lambda shape, dt: torch.zeros(shape, dtype=dt, device=device, pin_memory=pin)
    return [new((B, H, tokens, D * c["bits"] // 8), torch.uint8), new((B, H, tokens // G, D), METAS[c["meta"]]),
            new((B, H, tokens // G, D), METAS[c["meta"]])]


def _value_cache(c, tokens, device="cuda", pin=False):
    B, H, G = c["batch"], c["kv_heads"], c["group"]
    new = lambda shape, dt: torch.zeros(shape, dtype=dt, device=device, pin_memory=pin)
    return [new((B, H, tokens, D * c["bits"] // 8), torch.uint8), new((B, H, tokens, D // G), METAS[c["meta"]]),
            new((B, H, tokens, D // G), METAS[c["meta"]])]


def _pack(x, codes, scales, zeros, bits, dim):
    """Round-to-nearest groups of x (grouped along `dim`) as packed codes and their grids: a filled cache for the readers,
    made without the library so that their inputs depend on the seed alone."""
    lo, hi = x.amin(dim, keepdim=True), x.amax(dim, keepdim=True)
    scale = ((hi - lo) / (2 ** bits - 1)).to(scales.dtype)
    zero = lo.to(zeros.dtype)
    c = ((x - zero.float()) / scale.float()).round_().clamp_(0, 2 ** bits - 1).to(torch.uint8)
    scales.copy_(scale.view(scales.shape))
    zeros.copy_(zero.view(zeros.shape))
    c = c.view(*codes.shape, 8 // bits)
    out = c[..., 0].clone()
    for i in range(1, 8 // bits):
        out |= c[..., i] << (bits * i)
    codes.copy_(out)


def _filled_cache(c, g):
    B, H, T, G, bits = c["batch"], c["kv_heads"], c["tokens"], c["group"], c["bits"]
    k, v, outl = _key_cache(c, T), _value_cache(c, T), _outliers(H, g)
    for b in range(B):
        x = torch.randn((H, T, D), generator=g, device="cuda") * outl[:, None, :]
        _pack(x.view(H, T // G, G, D), k[0][b].view(H, T // G, G, -1), k[1][b], k[2][b], bits, 2)
        x = torch.randn((H, T, D), generator=g, device="cuda")
        _pack(x.view(H, T, D // G, G), v[0][b].view(H, T, D // G, -1), v[1][b], v[2][b], bits, 3)
    return k, v


def prepare(case, seed):
    c = dict(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + 17)
    B, H, T, dt = c["batch"], c["kv_heads"], c["tokens"], DTYPES[c["dtype"]]
    s = dict(case=c)
    if c["kind"] in ("prefill", "host"):
        s["q"] = _queries(c, g)
        s["k"] = _normal((B, H, T, D), g, dt, _outliers(H, g))
        s["v"] = _normal((B, H, T, D), g, dt)
        s["x0"] = torch.randn((D, c["rank"]), generator=g, device="cuda", dtype=torch.float64) if c["step1"] == "power" else None
        s["sub"] = sq.Subspace(H, D)
        if c["kind"] == "prefill":
            s["kc"], s["vc"] = _key_cache(c, T), _value_cache(c, T)
        else:
            for name in ("q", "k", "v", "x0"):
                if s[name] is not None:
                    s[name] = s[name].cpu().pin_memory()
            s["kc"], s["vc"] = _key_cache(c, T, "cpu", True), _value_cache(c, T, "cpu", True)
            n = sq.squat_write_path_workspace_bytes(dt, B, c["q_heads"], H, T, D, c["bits"], c["group"])
            s["ws"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    elif c["kind"] == "window":
        c["prompt"] = 1024                       # the prompt behind the update matrices that the window uses
        s["k"] = _normal((B, H, T, D), g, dt, _outliers(H, g))
        s["v"] = _normal((B, H, T, D), g, dt)
        s["sub"] = sq.Subspace(H, D)
        sq.squat_build_subspace(s["sub"], _queries(c, g), c["rank"], LAMBDA, c["block"])
        s["kc"], s["vc"] = _key_cache(c, c["cache"]), _value_cache(c, c["cache"])
        G, at = c["group"], c["cache"] - T       # the last window of the cache
        s["kw"] = [s["kc"][0][:, :, at:], s["kc"][1][:, :, at // G:], s["kc"][2][:, :, at // G:]]
        s["vw"] = [x[:, :, at:] for x in s["vc"]]
    else:
        s["kc"], s["vc"] = _filled_cache(c, g)
        if c["kind"] == "readback":
            s["out"] = [torch.empty((B, H, T, D), dtype=dt, device="cuda") for _ in range(2)]
        else:
            R, Hq = c["residual"], c["q_heads"]
            s["q"] = _normal((B, Hq, D), g, dt)
            s["k_res"] = _normal((B, H, R, D), g, dt, _outliers(H, g)) if R else None
            s["v_res"] = _normal((B, H, R, D), g, dt) if R else None
            s["out"] = torch.empty((B, Hq, D), dtype=torch.float32, device="cuda")
            n = sq.squat_decode_attention_workspace_bytes(B, Hq, T)
            s["ws"] = torch.empty(n, dtype=torch.uint8, device="cuda")
            if c["rope"]:
                s["positions"] = T + 128
                s["table"] = sq.squat_rope_table(s["positions"]).cuda()
    return s


# --------------------------------------------------------------------------------------------------------------- run
def run(s):
    c = s["case"]
    bits, group = c["bits"], c["group"]
    if c["kind"] == "prefill":
        if s["x0"] is None:
            sq.squat_build_subspace(s["sub"], s["q"], c["rank"], LAMBDA, c["block"])
        else:
            sq.squat_build_subspace_power(s["sub"], s["q"], c["rank"], LAMBDA, s["x0"], 2, c["block"])
        sq.squat_quantize_keys(s["sub"], s["k"], bits, group, *s["kc"])
        sq.squat_quantize_values(s["v"], bits, group, *s["vc"])
        return s["kc"], s["vc"]
    if c["kind"] == "window":
        H, L = c["kv_heads"], c["cache"]
        sq.squat_quantize_keys(s["sub"], s["k"], bits, group, *s["kw"], out_stride_b=H * L, out_stride_h=L)
        sq.squat_quantize_values(s["v"], bits, group, *s["vw"], out_stride_b=H * L, out_stride_h=L)
        return s["kw"], s["vw"]
    if c["kind"] == "attend":
        if c["rope"]:
            sq.squat_decode_attention_pre_rope(s["q"], *s["kc"], *s["vc"], c["kv_heads"], c["tokens"], bits, group, s["out"],
                                               s["ws"], s["table"], s["positions"], 0, s["k_res"], s["v_res"])
        else:
            sq.squat_decode_attention(s["q"], *s["kc"], *s["vc"], c["kv_heads"], c["tokens"], bits, group, s["out"], s["ws"],
                                      s["k_res"], s["v_res"])
        return s["out"]
    if c["kind"] == "readback":
        dims = (c["batch"], c["kv_heads"], c["tokens"], D, bits, group)
        sq.squat_dequantize(sq.SQUAT_KEYS, *s["kc"], *dims, s["out"][0])
        sq.squat_dequantize(sq.SQUAT_VALUES, *s["vc"], *dims, s["out"][1])
        return s["out"]
    sq.squat_write_path_host(s["sub"], s["q"], s["k"], s["v"], c["rank"], LAMBDA, c["block"], bits, group, *s["kc"], *s["vc"],
                             s["ws"], start_block=s["x0"])
    return s["kc"], s["vc"]


# -------------------------------------------------------------------------------------------------------------- work
def work(c):
    """Every input read once, every output written once; the operations of the method's own formulas."""
    B, H, T, G, bits = c["batch"], c["kv_heads"], c["tokens"], c["group"], c["bits"]
    size, msize, n = DTYPES[c["dtype"]].itemsize, METAS[c["meta"]].itemsize, c["batch"] * c["kv_heads"] * c["tokens"]
    packed = n * (2 * D * bits // 8 + 2 * msize * D // G + 2 * msize * D // G)          # both caches, codes and grids
    if c["kind"] in ("prefill", "window", "host"):
        g = c["block"]
        update = D * (D - g) if g > 1 else min(D * (D - 1), 4 * c["rank"] * D)         # per key vector (dense or rank-r form)
        nbytes, flops = 2 * n * D * size + packed, n * update + 10 * n * D
        if c["kind"] != "window":
            rows = c["q_heads"] * T                                                    # one sample's prompt queries
            nbytes += rows * D * size
            r = c["rank"]
            step1 = 9 * D ** 3 if c["step1"] == "svd" else 2 * 2 * D * D * r + 4 * D * r * r
            flops += rows * D * (D + 1) + H * (step1 + D ** 3)                         # Gram, subspace, update matrices
        else:
            nbytes += H * D * D * 4
        return {"bytes": nbytes, "flops": flops}
    if c["kind"] == "attend":
        R, Hq = c["residual"], c["q_heads"]
        nbytes = packed + 2 * B * H * R * D * size + B * Hq * D * (size + 4)
        return {"bytes": nbytes, "flops": 4 * B * Hq * (T + R) * D}
    return {"bytes": packed + 2 * n * D * size, "flops": 4 * n * D}


def tolerance(c):
    if c["kind"] == "readback":
        return "exact"                           # one rounding of an exact value
    if c["kind"] == "attend":
        return {"rel": 2e-5, "max": 4e-4}        # 32-bit scores and sums over up to 32768 tokens, with cancellation
    # A corrected key that lies on a rounding tie (within 1e-5 of a grid step) may go either way, and with it the later
    # channels of its token and, through the shared minimum and maximum, of its group.
    return {"rel": 3e-3, "max": 0.9, "differ": 5e-3}
