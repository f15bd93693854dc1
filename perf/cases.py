"""What a user of this library has it do, as cases that can be timed and compared.

Every case is one call (or one decode step's calls) through the public entry points of
`paper_2503_01586_b200.binding` on synthetic inputs of the library's own layer shapes
(`paper_2503_01586_b200.inputs`).  A case is a dict of plain values:

  kind    "step"    one decode step of a layer: elitekv_decode_step (append + query preparation +
                    attention) on device buffers that a serving loop keeps
          "host"    the same step from host arrays to a host result, replayed from a CUDA graph
                    (DecodeStepRunner)
          "hidden"  a decode step that starts from the hidden states: elitekv_project_append, then
                    elitekv_absorb_query and elitekv_decode
          "rows"    several query rows per sequence (draft tokens of speculative decoding, a chunk
                    of a prefill): elitekv_absorb_query + elitekv_attend_rows
          "append"  prefill: keys and latents of whole prompts rotated into the cache
          "project" prefill from the hidden states: projection fused with the append
          "search"  RoPElite calibration (Algorithm 1) over the heads of a layer
  layer   name of the layer shape: a key of LAYERS
  B, ctx, ctx_lo, paged, lens_seed
          sequences, longest context, shortest context (== ctx: all equal), cache layout, seed of
          the ragged lengths (so that a case does the same work whatever its inputs' seed is)
"""
from __future__ import annotations

import math
from dataclasses import replace

import torch

from paper_2503_01586_b200 import binding as ek
from paper_2503_01586_b200 import inputs as gen

DEVICE = "cuda"

# layer shapes: the repository's benchmark configurations (batch and context come from the case)
LAYERS = {
    "tiny": gen.TINY,
    "7b-75": gen.LLAMA7B_75,
    "13b-75": gen.LLAMA13B_75,
    "7b-50": gen.SWEEP_50,
    "7b-87.5": gen.SWEEP_875,
    "7b-75-slrd": gen.SWEEP_75_SLRD,
}


def _attend(name, kind, layer, B, ctx, ctx_lo=None, paged=False, lens_seed=0, **more):
    case = {"kind": kind, "layer": layer, "B": B, "ctx": ctx, "ctx_lo": ctx if ctx_lo is None else ctx_lo,
            "paged": paged, "lens_seed": lens_seed, **more}
    return case if name is None else {"name": name, **case}


def listed():
    return [
        # the smallest model configuration, one sequence: a step is launches and latency only
        _attend("tiny-b1-ctx256", "step", "tiny", 1, 256),
        # one interactive user of a 7B layer, odd context, inputs and result on the host
        _attend("7b-75-host-b1-ctx1999", "host", "7b-75", 1, 1999),
        # the headline: a serving batch at moderate context
        _attend("7b-75-b16-ctx4096", "step", "7b-75", 16, 4096),
        # continuous batching: ragged lengths up to 32768 over a paged cache with shuffled pages
        _attend("7b-75-paged-b64-ragged", "step", "7b-75", 64, 32768, ctx_lo=1024, paged=True, lens_seed=1003),
        # 13B layer (40 heads), long contexts: the most cache bytes among the dense batches
        _attend("13b-75-b32-ctx16384", "step", "13b-75", 32, 16384),
        # the other two compression ratios at the sweep's batch and context; the narrow one starts
        # from the hidden states, so that its step holds the projection at decode size
        _attend("7b-50-b32-ctx8192", "step", "7b-50", 32, 8192),
        _attend("7b-87.5-hidden-b32-ctx8192", "hidden", "7b-87.5", 32, 8192),
        # separated key and value latents (S-LRD)
        _attend("7b-75-slrd-b32-ctx8192", "step", "7b-75-slrd", 32, 8192),
        # four draft tokens per sequence, ragged contexts
        _attend("7b-75-rows4-b16-ragged", "rows", "7b-75", 16, 4096, ctx_lo=1024, lens_seed=7, rows=4),
        # 32 prompts of 4096 tokens enter the cache
        _attend("7b-75-append-32x4096", "append", "7b-75", 32, 4096),
        # one prompt of 4096 hidden states is projected into the cache
        _attend("7b-75-project-4096", "project", "7b-75", 1, 4096),
        # calibration of one layer: 32 heads, 2048 tokens, 8 chunks chosen
        {"name": "search-32x2048-r8", "kind": "search", "heads": 32, "n": 2048, "d_h": 128, "r": 8},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


MAX_CACHE_BYTES = 4.4e9      # the ragged listed case


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "host", "hidden", "rows", "append", "project", "search"])
    if kind == "search":
        d_h = rng.choice([64, 128])
        n, r = _log_int(rng, 128, 2048), rng.randint(1, 16)
        # no more pair sums than the listed search
        heads = min(_log_int(rng, 4, 64), int(32 * (2048 / n) ** 2 * (8 / r) * (128 / d_h)))
        return {"kind": kind, "heads": max(heads, 1), "n": n, "d_h": d_h, "r": r}
    if kind in ("append", "project"):
        layer = rng.choice(["7b-75", "13b-75", "7b-50", "7b-87.5", "7b-75-slrd"])
        B = _log_int(rng, 1, 32)
        tokens = _log_int(rng, B, 65536 if kind == "append" else 16384)
        ctx = max(1, tokens // B)
        return _attend(None, kind, layer, B, ctx, ctx_lo=max(1, ctx // 2), paged=rng.random() < 0.5,
                       lens_seed=rng.randrange(1 << 20))
    layer = rng.choice(["7b-75", "7b-75", "7b-75", "13b-75", "7b-50", "7b-87.5", "7b-75-slrd"])
    if kind == "step" and rng.random() < 0.15:
        return _attend(None, kind, "tiny", _log_int(rng, 1, 16), _log_int(rng, 16, 2048),
                       paged=rng.random() < 0.5, lens_seed=rng.randrange(1 << 20))
    B = _log_int(rng, 1, 64)
    most = MAX_CACHE_BYTES / (2 * LAYERS[layer].cache_elems_per_token * B)
    ctx = _log_int(rng, 64, int(min(32768, most)))
    more = {}
    if kind == "rows":
        more["rows"] = rng.choice([2, 3, 4, 5, 8])
        ctx = max(64, ctx // 4)
    ragged = rng.random() < 0.6
    return _attend(None, kind, layer, B, ctx, ctx_lo=max(16, ctx // 8) if ragged else ctx,
                   paged=rng.random() < 0.5, lens_seed=rng.randrange(1 << 20), **more)


# ------------------------------------------------------------------------------- preparation
def _workload(case, seed):
    w = LAYERS[case["layer"]]
    return replace(w, name="case", B=case["B"], ctx=case["ctx"], ctx_lo=None, paged=case["paged"], seed=seed)


def _lengths(case):
    """int32 [B], the token being decoded included: fixed by the case."""
    if case["ctx_lo"] == case["ctx"]:
        return torch.full((case["B"],), case["ctx"], dtype=torch.int32)
    g = torch.Generator().manual_seed(case["lens_seed"])
    return torch.randint(case["ctx_lo"], case["ctx"] + 1, (case["B"],), generator=g).to(torch.int32)


def _normal(shape, seed, std=1.0):
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    out = torch.empty(shape, dtype=torch.bfloat16, device=DEVICE)
    flat = out.view(-1)
    for lo in range(0, flat.numel(), 1 << 28):
        hi = min(flat.numel(), lo + (1 << 28))
        flat[lo:hi] = torch.randn(hi - lo, generator=g, device=DEVICE) * std
    return out


def _layer_and_cache(case, seed, w, lens, projection=False, filled=True):
    """The layer handle and a cache that holds `lens` tokens per sequence.  Rotated keys and latents
    are N(0, 1): the law of x W for x ~ N(0, 1) and W ~ N(0, 1/d), which a rotation leaves alone."""
    W_uk, W_uv = gen.up_projections(w, DEVICE)
    if w.d_ck:
        W_uk, W_uv = W_uk[:w.d_ck].contiguous(), W_uv[w.d_ck:].contiguous()
    rope_w, max_ctx = w.n_h * 2 * w.r, int(lens.max())
    more = {}
    if projection:
        more = {"W_ke": _normal((w.d, rope_w), seed * 7 + 11, (1.0 / w.d) ** 0.5),
                "W_down": _normal((w.d, w.d_c), seed * 7 + 12, (1.0 / w.d) ** 0.5)}
    layer = ek.Layer(w.n_h, w.d_h, w.r, w.d_c, gen.elite_index_sets(w), W_uk, W_uv, max_ctx + 1,
                     rope_base=w.rope_base, d_ck=w.d_ck, **more)
    table = None
    if w.paged:
        table, num_pages = gen.page_table(w, lens, headroom_tokens=0)
        rows, table = num_pages * w.page_size, table.to(DEVICE)
    else:
        rows = w.B * max_ctx
    if filled:
        rope, latent = _normal((rows, rope_w), seed * 7 + 13), _normal((rows, w.d_c), seed * 7 + 14)
    else:
        rope = torch.zeros((rows, rope_w), dtype=torch.bfloat16, device=DEVICE)
        latent = torch.zeros((rows, w.d_c), dtype=torch.bfloat16, device=DEVICE)
    cache = ek.make_cache(rope, latent, n_seqs=w.B, max_ctx=max_ctx, page_table=table, page_size=w.page_size)
    return {"layer": layer, "cache": cache, "rope": rope, "latent": latent, "table": table}


def _prompt_tokens(lens):
    """seq_id and pos of whole prompts, token after token."""
    seq = torch.repeat_interleave(torch.arange(lens.numel(), dtype=torch.int32), lens.long())
    pos = torch.cat([torch.arange(int(n), dtype=torch.int32) for n in lens])
    return seq.to(DEVICE), pos.to(DEVICE)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "search":
        H, n, d_h = case["heads"], case["n"], case["d_h"]
        # every head has its own preference among the frequencies: graded energies per chunk
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        scale = torch.exp(0.4 * torch.randn((H, 1, d_h // 2, 1), generator=g, device=DEVICE))
        scale = scale.expand(H, 1, d_h // 2, 2).reshape(H, 1, d_h)
        s["Q"], s["K"] = ((torch.randn((H, n, d_h), generator=g, device=DEVICE) * scale).to(torch.bfloat16)
                          for _ in range(2))
        s["r"] = case["r"]
        s["ws"] = torch.empty(ek.elitekv_ropelite_workspace_size(H, n, d_h), dtype=torch.uint8, device=DEVICE)
        return s
    w, lens = _workload(case, seed), _lengths(case)
    B = w.B
    if kind in ("append", "project"):
        s.update(_layer_and_cache(case, seed, w, lens, projection=kind == "project", filled=False))
        s["seq"], s["pos"] = _prompt_tokens(lens)
        T = s["seq"].numel()
        if kind == "append":
            s["k_e"], s["c"] = _normal((T, w.n_h, w.r, 2), seed * 7 + 15), _normal((T, w.d_c), seed * 7 + 16)
        else:
            s["x"] = _normal((T, w.d), seed * 7 + 17)
        return s
    s.update(_layer_and_cache(case, seed, w, lens, projection=kind == "hidden"))
    layer = s["layer"]
    new = {"seq": torch.arange(B, dtype=torch.int32), "pos": lens - 1, "lens": lens}
    if kind == "host":
        run = s["runner"] = ek.DecodeStepRunner(layer, s["cache"], B, DEVICE)
        k_e, c = gen.tokens(w, B, "cpu")
        for name, value in (("k_e", k_e), ("c", c), ("q", gen.queries(w)), ("seq_id", new["seq"]),
                            ("pos", new["pos"]), ("lens", lens)):
            run.host[name].copy_(value.view(run.host[name].shape))
        return s
    s.update({k: v.to(DEVICE) for k, v in new.items()})
    m = s["m"] = case.get("rows", 1)
    s["q"] = _normal((B * m, w.n_h, w.d_h), seed * 7 + 18)
    s["q_rope"] = torch.empty((B * m, w.n_h, 2 * w.r), dtype=torch.bfloat16, device=DEVICE)
    s["q_abs"] = torch.empty((B * m, w.n_h, layer.kw), dtype=torch.bfloat16, device=DEVICE)
    s["out"] = torch.empty((B, m, w.n_h, w.d_h) if kind == "rows" else (B, w.n_h, w.d_h),
                           dtype=torch.bfloat16, device=DEVICE)
    if kind == "rows":
        s["q_pos"] = (s["lens"].view(B, 1) - m + torch.arange(m, device=DEVICE).view(1, m)).to(torch.int32).view(-1)
        size = ek.elitekv_attend_rows_workspace_size(layer, B, m)
    else:
        size = ek.elitekv_decode_workspace_size(layer, B)
    s["ws"] = torch.empty(size, dtype=torch.uint8, device=DEVICE)
    if kind == "hidden":
        s["x"] = _normal((B, w.d), seed * 7 + 17)
    else:
        s["k_e"], s["c"] = _normal((B, w.n_h, w.r, 2), seed * 7 + 15), _normal((B, w.d_c), seed * 7 + 16)
    return s


# ------------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "search":
        idx, trace = ek.elitekv_ropelite_search(s["Q"], s["K"], s["r"], trace=True, workspace=s["ws"])
        return {"elite_idx": idx, "distances": trace}
    layer, cache = s["layer"], s["cache"]
    planes = {"rope": s["rope"], "latent": s["latent"]}
    if kind == "append":
        ek.elitekv_append(layer, cache, s["k_e"], s["c"], s["seq"], s["pos"])
        return planes
    if kind == "project":
        ek.elitekv_project_append(layer, cache, s["x"], s["seq"], s["pos"])
        return planes
    if kind == "host":
        return {"out": s["runner"].run(), **planes}
    if kind == "step":
        ek.elitekv_decode_step(layer, cache, s["k_e"], s["c"], s["seq"], s["pos"], s["q"], s["lens"],
                               s["q_rope"], s["q_abs"], s["ws"], s["out"])
    elif kind == "hidden":
        ek.elitekv_project_append(layer, cache, s["x"], s["seq"], s["pos"])
        ek.elitekv_absorb_query(layer, s["q"], s["pos"], s["q_rope"], s["q_abs"])
        ek.elitekv_decode(layer, cache, s["q_rope"], s["q_abs"], s["lens"], s["ws"], s["out"])
    else:
        ek.elitekv_absorb_query(layer, s["q"], s["q_pos"], s["q_rope"], s["q_abs"])
        ek.elitekv_attend_rows(layer, cache, s["q_rope"], s["q_abs"], s["lens"], s["m"], s["ws"], s["out"])
    outs = {"out": s["out"], "q_rope": s["q_rope"], "q_abs": s["q_abs"]}
    return outs if kind == "rows" else {**outs, **planes}


# ------------------------------------------------------------------------------- what it takes
def work(case):
    """Bytes: cache rows, weights, inputs and outputs, each once.  Flops: the two contractions over
    the cache (absorbed form), the absorption, the up-projection and the projections."""
    if case["kind"] == "search":
        H, n, half, r = case["heads"], case["n"], case["d_h"] // 2, case["r"]
        pairs = H * n * (n + 1) // 2
        # D_i = a_i (cos - 1) - b_i sin once per pair and chunk (9), then one |R - D_j| sum (3) per
        # pair, chunk and round
        return {"bytes": 2 * 2 * H * n * case["d_h"] + 4 * r * H * (half + 1), "flops": pairs * half * (9 + 3 * r)}
    w = LAYERS[case["layer"]]
    n, B, m = int(_lengths(case).sum()), case["B"], case.get("rows", 1)
    kw, vw = (w.d_ck, w.d_c - w.d_ck) if w.d_ck else (w.d_c, w.d_c)
    row, proj = 2 * w.cache_elems_per_token, 2 * w.d * w.cache_elems_per_token
    if case["kind"] == "append":
        return {"bytes": n * (2 * row + 8), "flops": n * w.n_h * w.r * 6}
    if case["kind"] == "project":
        return {"bytes": n * (2 * w.d + row + 8) + proj, "flops": n * proj}
    weights = 2 * w.n_h * (w.d_nope * kw + w.d_h * vw)
    q_bytes = 2 * B * m * w.n_h * (2 * w.d_h + 2 * w.r + kw)      # q, out, q_rope, q_abs
    bytes_ = n * row + weights + q_bytes
    flops = m * (n * w.n_h * (4 * w.r + 2 * kw + 2 * vw) + 2 * B * w.n_h * (w.d_nope * kw + w.d_h * vw))
    if case["kind"] == "hidden":
        bytes_ += proj + 2 * B * w.d + B * row
        flops += B * proj
    elif case["kind"] != "rows":
        bytes_ += 2 * B * row
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    if case["kind"] == "append":
        return "exact"            # every product and sum of the rotation is rounded separately: bits are fixed
    if case["kind"] == "search":
        # fp32 sums over up to n^2 / 2 pairs in another order; a choice between two chunks whose
        # distances agree to the last bits may fall the other way
        return {"rel": 1e-5, "max": 5e-5, "differ": 0.01}
    if case["kind"] == "project":
        # one rounding to bf16 of fp32 sums: 1.7e-3 (largest 4e-3) against float64
        return {"rel": 6e-3, "max": 2e-2}
    # bf16 queries, cache and probabilities, fp32 sums: 2.5e-3 (largest 8e-3) against float64
    return {"rel": 1e-2, "max": 4e-2}
