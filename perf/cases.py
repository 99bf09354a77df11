"""Performance cases: the decode steps of a GQLA attention layer and the one-shot cache expansion, through the
package's public entry points (`GqlaDecoder` and the binding's FP8 calls).

Dimensions are the canonical (h_q, g, d_h, r_kv, d_h^R) = (128, 8, 128, 512, 64) and the LLaMA-3-8B-shaped h_q = 32;
`draw` adds 64 heads and the 28 heads in 4 groups of the parity tests.  A decode step is served the way bench.py
serves it: the call chain is captured once into a CUDA graph (`GqlaDecoder.capture`) and replayed per step.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2605_15250_b200 import binding as B
from paper_2605_15250_b200.decoder import GqlaDecoder

D_H, R_KV, D_R = 128, 512, 64
SCALE = 1.0 / math.sqrt(D_H + D_R)
TILE = 128  # rows the balanced plan counts in

# E4M3 plane scales of N(0, 1) data (about 5.6 standard deviations at the largest code)
FP8_SCALE = 5.6 / 448.0


def _case(name, kind, h_q, batch, s_q, t_lo, t_hi, page=0, g=8):
    c = {"kind": kind, "h_q": h_q, "g": g, "batch": batch, "s_q": s_q, "t_lo": t_lo, "t_hi": t_hi, "page": page}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one user's chat, MQA-absorb path: a call of a few kernels over a short cache, all latency
        _case("absorb_one", "absorb", 128, 1, 1, 777, 777),
        # a full serving batch on the canonical shape, one piece per sequence (bench.py's workload)
        _case("absorb_batch", "absorb", 128, 64, 1, 4096, 4096),
        # the same with two draft tokens per step and the ragged lengths of continuous batching
        _case("absorb_mtp_ragged", "absorb", 128, 48, 2, 1000, 9001),
        # LLaMA-3-8B-shaped conversion, large ragged batch
        _case("absorb_llama", "absorb", 32, 128, 1, 512, 32768),
        # a few long documents: split-KV over the whole GPU and the merge of many pieces
        _case("absorb_long", "absorb", 128, 4, 1, 131072, 131072),
        # one user's chat on the GQA path
        _case("gqa_one", "gqa", 128, 1, 1, 3001, 3001),
        # the serving batch on the GQA path with multi-token prediction
        _case("gqa_batch_mtp", "gqa", 128, 64, 2, 4096, 4096),
        # LLaMA-3-8B-shaped on the GQA path: the largest cache
        _case("gqa_llama", "gqa", 32, 128, 1, 512, 32768),
        # the serving batch over an E4M3 cache, both paths
        _case("absorb_fp8", "absorb_fp8", 128, 64, 1, 4096, 4096),
        _case("gqa_fp8_mtp", "gqa_fp8", 128, 64, 2, 4096, 4096),
        # continuous batching over a block-table cache with the 64-row blocks that latent-attention servers use
        _case("absorb_paged", "absorb_paged", 128, 32, 1, 300, 8000, page=64),
        # switching a prefilled batch from the absorb path to the GQA path
        _case("expand", "expand", 128, 50, 1, 3000, 5999),
    ]


def _log_int(rng: random.Random, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("absorb", "absorb", "gqa", "gqa", "absorb_fp8", "gqa_fp8", "absorb_paged", "gqa_paged", "expand"))
    h_q, g = rng.choice(((128, 8), (128, 8), (64, 8), (32, 8), (28, 4)))
    page = rng.choice((16, 32, 64, 128, 256)) if kind.endswith("paged") else 0
    s_q = 1 if kind == "expand" else rng.choice((1, 1, 2))
    rows = {"absorb": 1 << 20, "gqa": 1 << 21, "absorb_fp8": 1 << 20, "gqa_fp8": 1 << 20, "expand": 1 << 18}.get(kind, 1 << 18)
    t_hi = _log_int(rng, 100, min(131072, rows))
    batch = _log_int(rng, 1, max(1, min(128, rows // t_hi)))
    t_lo = t_hi if rng.random() < 0.4 else max(s_q, t_hi // rng.choice((2, 8, 64)))
    return _case("", kind, h_q, batch, s_q, t_lo, t_hi, page, g)


def _lengths(case):
    """The batch's lengths are the case's own: every seed draws other values for the same batch."""
    rng = random.Random("%d %d %d" % (case["batch"], case["t_lo"], case["t_hi"]))
    return [rng.randint(case["t_lo"], case["t_hi"]) for _ in range(case["batch"])]


def _normal(gen, shape, mul=1.0):
    out = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    flat = out.view(-1)
    for lo in range(0, flat.numel(), 1 << 28):
        part = flat[lo:lo + (1 << 28)]
        part.copy_(torch.randn(part.numel(), generator=gen, device="cuda", dtype=torch.float32).mul_(mul))
    return out


def _inputs(case, seed):
    """Queries, weights and latent cache rows (unit-variance scaled scores), the packed layout."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    lens = _lengths(case)
    b, s, h, g = case["batch"], case["s_q"], case["h_q"], case["g"]
    starts = [0]
    for t in lens[:-1]:
        starts.append(starts[-1] + t)
    return {
        "lens": lens, "starts": starts,
        "q": _normal(gen, (b, s, h, D_H + D_R)),
        "w_uk": _normal(gen, (g, R_KV, D_H), 1.0 / math.sqrt(R_KV)),
        "w_uv": _normal(gen, (g, R_KV, D_H), 1.0 / math.sqrt(R_KV)),
        "cache": _normal(gen, (sum(lens), R_KV + D_R)),
    }


def _paged(case, seed, x):
    """The cache scattered over a shuffled pool of pages, as after some time of serving, and its block table."""
    page, lens = case["page"], x["lens"]
    counts = [-(-t // page) for t in lens]
    order = list(range(sum(counts) + 3))
    random.Random(seed + 1).shuffle(order)
    table = torch.zeros((len(lens), max(counts)), dtype=torch.int32)
    at = 0
    for i, n in enumerate(counts):
        table[i, :n] = torch.tensor(order[at:at + n], dtype=torch.int32)
        at += n
    table = table.cuda()
    pool = torch.zeros((len(order) * page, R_KV + D_R), dtype=torch.bfloat16, device="cuda")
    for i, (t, s) in enumerate(zip(lens, x["starts"])):
        pos = torch.arange(t, device="cuda")
        pool[table[i, pos // page].long() * page + pos % page] = x["cache"][s:s + t]
    return pool, table


def _num_splits(case, lens, path, workers):
    """One piece per sequence where equal sequences fill the GPU by themselves (absorb path), else the balanced plan
    with as many slots as the longest sequence's share of the workers takes."""
    tiles = [-(-t // TILE) for t in lens]
    units = case["batch"] * (-(-case["s_q"] * case["h_q"] // 128))
    if path == "absorb" and min(lens) == max(lens) and units >= 0.8 * workers:
        return 1
    share = max(1, -(-sum(tiles) // max(workers, 1)))
    slots = -(-max(tiles) // share) + 1
    return -slots


def _fp8_absorb(dec, q_c, q_r, cache8, splits):
    """absorb_q -> quantize_rows -> decode -> up-projection over an E4M3 latent cache, in buffers of its own."""
    b, s, h = q_c.shape[:3]
    bf = {"dtype": torch.bfloat16, "device": "cuda"}
    f32 = {"dtype": torch.float32, "device": "cuda"}
    q_hat = torch.empty((b, s, h, R_KV + D_R), **bf)
    q8 = torch.empty(q_hat.shape, dtype=torch.uint8, device="cuda")
    q_scale = torch.empty((b, s, h), **f32)
    o_hat = torch.empty((b, s, h, R_KV), **bf)
    o_part = torch.empty((b, abs(splits), s, h, R_KV), **f32)
    lse_part = torch.empty((b, abs(splits), s, h), **f32)
    o = torch.empty((b, s, h, D_H), **bf)

    def step():
        B.gqla_absorb_q(dec.dims, q_c, q_r, dec.w_uk, q_hat)
        B.gqla_quantize_rows_e4m3(q_hat, R_KV, FP8_SCALE, FP8_SCALE, q8, q_scale)
        if splits == 1:
            B.gqla_decode_absorb_fp8_final(dec.dims, q8, q_scale, cache8, FP8_SCALE, dec.seq_start, dec.seqlens, SCALE,
                                           o_hat, None, dec.status)
            B.gqla_up_proj(dec.dims, o_hat, dec.w_uv, o)
            return o
        B.gqla_decode_absorb_fp8(dec.dims, q8, q_scale, cache8, FP8_SCALE, dec.seq_start, dec.seqlens, SCALE, splits,
                                 o_part, lse_part, dec.status)
        if abs(splits) <= 4:
            B.gqla_combine_up_proj(dec.dims, o_part, lse_part, dec.w_uv, o)
        else:
            B.gqla_combine_splits(o_part, lse_part, o_hat)
            B.gqla_up_proj(dec.dims, o_hat, dec.w_uv, o)
        return o
    return step


def _fp8_gqa(dec, q, planes, splits):
    b, s, h = q.shape[:3]
    f32 = {"dtype": torch.float32, "device": "cuda"}
    q8 = torch.empty(q.shape, dtype=torch.uint8, device="cuda")
    q_scale = torch.empty((b, s, h), **f32)
    o_part = torch.empty((b, abs(splits), s, h, D_H), **f32)
    lse_part = torch.empty((b, abs(splits), s, h), **f32)
    o = torch.empty((b, s, h, D_H), dtype=torch.bfloat16, device="cuda")

    def step():
        B.gqla_quantize_rows_e4m3(q, D_H, FP8_SCALE, FP8_SCALE, q8, q_scale)
        B.gqla_decode_gqa_fp8(dec.dims, q8, q_scale, *planes, FP8_SCALE, dec.seq_start, dec.seqlens, SCALE, splits,
                              o_part, lse_part, dec.status)
        B.gqla_combine_splits(o_part, lse_part, o)
        return o
    return step


def _quantize(t, width):
    out = torch.empty(t.shape, dtype=torch.uint8, device="cuda")
    B.gqla_quantize_cols_e4m3(t, width, FP8_SCALE, FP8_SCALE, out)
    return out


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, lens = case["kind"], x["lens"]
    seqlens = torch.tensor(lens, dtype=torch.int32, device="cuda")
    seq_start = torch.tensor(x["starts"], dtype=torch.int64, device="cuda")
    cache, table, page = x["cache"], None, case["page"]
    if page:
        cache, table = _paged(case, seed, x)
        seq_start = None
    dec = GqlaDecoder(case["h_q"], case["g"], D_H, R_KV, D_R, x["w_uk"], x["w_uv"], cache, seq_start, seqlens, SCALE,
                      block_table=table, page_size=page)
    state = {"dec": dec}
    if kind == "expand":
        return state
    path = kind.split("_")[0]
    workers = B.gqla_balanced_workers(dec.dims, torch.bfloat16, case["s_q"], path)
    splits = _num_splits(case, lens, path, workers)
    q = x["q"]
    if path == "gqa":
        dec.expand_cache()
    q_c, q_r = q[..., :D_H].contiguous(), q[..., D_H:].contiguous()
    if kind == "absorb_fp8":
        step, args = _fp8_absorb(dec, q_c, q_r, _quantize(cache, R_KV), splits), ()
    elif kind == "gqa_fp8":
        planes = [_quantize(dec.k_c, D_H), _quantize(dec.v, D_H), _quantize(dec.k_r, D_R)]
        dec.k_c = dec.v = dec.k_r = None
        step, args = _fp8_gqa(dec, q, planes, splits), ()
    elif path == "absorb":
        step, args = dec.absorb_step, (q_c, q_r, splits)
    else:
        step, args = dec.gqa_step, (q, splits)
    # the captured graph reads these tensors on every replay: a program keeps them as long as the graph
    state["step"], state["args"] = step, args
    state["replay"], state["out"] = dec.capture(step, *args)
    return state


def run(state):
    if "replay" in state:
        state["replay"]()
        return state["out"]
    dec = state["dec"]
    dec.expand_cache()
    return dec.k_c, dec.v


def work(case):
    """Cache once, queries, weights and outputs once; the two contractions of the path (Eqs. (mqa), (mha))."""
    rows = sum(_lengths(case))
    h, g, n_q = case["h_q"], case["g"], case["batch"] * case["s_q"] * case["h_q"]
    weights = 2 * g * R_KV * D_H * 2
    if case["kind"] == "expand":
        return {"bytes": rows * 2 * (R_KV + 2 * g * D_H) + weights, "flops": 2.0 * rows * R_KV * 2 * g * D_H}
    size = 1 if case["kind"].endswith("fp8") else 2
    q_bytes = n_q * 2 * (D_H + D_R + D_H)
    if case["kind"].startswith("absorb"):
        return {"bytes": rows * size * (R_KV + D_R) + q_bytes + weights,
                "flops": 2.0 * rows * h * case["s_q"] * (2 * R_KV + D_R) + 4.0 * n_q * R_KV * D_H}
    return {"bytes": rows * size * (2 * g * D_H + D_R) + q_bytes, "flops": 2.0 * rows * h * case["s_q"] * (2 * D_H + D_R)}


def tolerance(case):
    """bf16: probabilities, latent queries and outputs are rounded to 8 bits; E4M3: probabilities keep 4 bits."""
    if case["kind"] == "expand":
        return {"rel": 2e-3, "max": 2e-2}
    if case["kind"].endswith("fp8"):
        return {"rel": 3e-2, "max": 0.5}
    return {"rel": 1e-2, "max": 0.1}


def _e4m3(t):
    """What a value is after the E4M3 cache's rounding, in 64 bits."""
    code = (t.float() * (1.0 / torch.tensor(FP8_SCALE, dtype=torch.float32))).clamp(-448, 448).to(torch.float8_e4m3fn)
    return code.double() * FP8_SCALE


def exact(case, seed):
    """The attention equations in 64 bits, one sequence after the other.  On the GQA path the keys and values are
    rounded to the cache's storage type, as the expanded cache a program has in hand is; on both paths E4M3
    caches hold rounded values and the queries are taken unrounded."""
    x = _inputs(case, seed)
    h, g, s_q = case["h_q"], case["g"], case["s_q"]
    w_uk, w_uv, q = x["w_uk"].double(), x["w_uv"].double(), x["q"].double()
    per = h // g
    fp8 = case["kind"].endswith("fp8")
    if case["kind"] == "expand":
        out = [torch.empty((sum(x["lens"]), g, D_H), dtype=torch.float64, device="cuda") for _ in range(2)]
        for lo in range(0, out[0].shape[0], 1 << 15):
            c = x["cache"][lo:lo + (1 << 15), :R_KV].double()
            for o, w in zip(out, (w_uk, w_uv)):
                o[lo:lo + (1 << 15)] = torch.einsum("nr,grd->ngd", c, w)
        return tuple(out)
    out = torch.empty((case["batch"], s_q, h, D_H), dtype=torch.float64, device="cuda")
    for b, (t, s) in enumerate(zip(x["lens"], x["starts"])):
        rows = x["cache"][s:s + t]
        c, k_r = rows[:, :R_KV].double(), rows[:, R_KV:].double()
        qb = q[b].view(s_q, g, per, D_H + D_R)
        if case["kind"].startswith("absorb"):
            if fp8:
                c, k_r = _e4m3(rows[:, :R_KV]), _e4m3(rows[:, R_KV:])
            latent = torch.einsum("sgpd,grd->sgpr", qb[..., :D_H], w_uk)
            scores = torch.einsum("sgpr,nr->sgpn", latent, c)
        else:
            planes = [torch.einsum("nr,grd->gnd", c, w).to(torch.bfloat16) for w in (w_uk, w_uv)]
            k_c, v = (_e4m3(p) if fp8 else p.double() for p in planes)
            k_r = _e4m3(rows[:, R_KV:]) if fp8 else k_r
            scores = torch.einsum("sgpd,gnd->sgpn", qb[..., :D_H], k_c)
        scores = (scores + torch.einsum("sgpd,nd->sgpn", qb[..., D_H:], k_r)) * SCALE
        for p in range(s_q):  # the step's later tokens are hidden from its earlier ones
            scores[p, :, :, t - (s_q - 1 - p):] = -math.inf
        prob = torch.softmax(scores, dim=-1)
        if case["kind"].startswith("absorb"):
            o = torch.einsum("sgpr,grd->sgpd", torch.einsum("sgpn,nr->sgpr", prob, c), w_uv)
        else:
            o = torch.einsum("sgpn,gnd->sgpd", prob, v)
        out[b] = o.reshape(s_q, h, D_H)
    return out
