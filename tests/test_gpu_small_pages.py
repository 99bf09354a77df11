"""Paged decode calls that the tensor-core kernels fetch in boxes within a page: pages of a multiple of 16 rows that are no
multiple of the 128-row tile, and pieces that start inside a tile."""
import numpy as np
import pytest
import torch

from paper_2605_15250_b200 import binding as B
from paper_2605_15250_b200 import build as gbuild
from paper_2605_15250_b200 import synth

pytestmark = pytest.mark.gpu

CANON = dict(h_q=128, g=8, d_h=128, r_kv=512, d_r=64)
LLAMA = dict(CANON, h_q=32)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    gbuild.build()
    assert torch.cuda.is_available()
    B.lib()
    B.set_policy(B.POLICY_AUTO)
    yield
    B.set_policy(B.POLICY_AUTO)


def _absorb(bd, w, q_hat, cache, table, page, sl, S, status, scale=None):
    o = torch.zeros((w.batch, abs(S), w.s_q, w.h_q, w.r_kv), device="cuda")
    lse = torch.full((w.batch, abs(S), w.s_q, w.h_q), float("nan"), device="cuda")
    B.gqla_decode_absorb_paged(bd, q_hat, cache, table, page, sl, w.scale if scale is None else scale, S, o, lse, status)
    return o, lse


def _gqa(bd, w, q, k_c, v, k_r, table, page, sl, S, status, scale=None):
    o = torch.zeros((w.batch, abs(S), w.s_q, w.h_q, w.d_h), device="cuda")
    lse = torch.full((w.batch, abs(S), w.s_q, w.h_q), float("nan"), device="cuda")
    B.gqla_decode_gqa_paged(bd, q, k_c, v, k_r, table, page, sl, w.scale if scale is None else scale, S, o, lse, status)
    return o, lse


@pytest.mark.parametrize("dims", [CANON, LLAMA, dict(LLAMA, h_q=16)])
@pytest.mark.parametrize("page,S,s_q", [(16, 1, 1), (16, -3, 2), (32, -3, 1), (48, 2, 1), (64, 1, 2), (64, -4, 1), (192, 3, 1), (128, 2, 1)])
@pytest.mark.parametrize("fill", [float("nan"), float("inf")])
def test_rows_that_no_sequence_owns_may_hold_anything(dims, page, S, s_q, fill):
    """NaN or infinity in every row of the pool behind a sequence's end and in the spare pages: bit for bit what a pool
    of zeros gives.  Ends at every remainder of eight rows, at the edges of boxes, tiles and pages."""
    seqlens = np.array([*range(1, 18), 0, 31, 33, 62, 63, 64, 65, 71, 100, 127, 128, 129, 190, 193, 257, 300], dtype=np.int32)
    w = synth.Workload("tails", batch=len(seqlens), s_q=s_q, dtype="bf16", seed=301, **dims)
    x = synth.make_inputs(w, seqlens=seqlens, q_gain=4.0)
    bd = B.make_dims(w.h_q, w.g, w.d_h, w.r_kv, w.d_r)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    sl = x["seqlens"].cuda()
    zero, table = synth.to_paged(x["cache"], x["seq_start"], seqlens, page, seed=302, fill=0.0)
    owned, _ = synth.to_paged(torch.ones(x["cache"].shape[0], 1), x["seq_start"], seqlens, page, seed=302, fill=0.0)
    zero, table, free = zero.cuda(), table.cuda(), (owned[:, 0] == 0).cuda()
    q = torch.cat([x["q_c"], x["q_r"]], -1).contiguous().cuda()
    q_hat = torch.empty((w.batch, s_q, w.h_q, w.d_abs), dtype=torch.bfloat16, device="cuda")
    B.gqla_absorb_q(bd, x["q_c"].cuda(), x["q_r"].cuda(), x["w_uk"].cuda(), q_hat)
    k_c, v = (torch.empty((zero.shape[0], w.g, w.d_h), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    B.gqla_expand_cache(bd, zero, x["w_uk"].cuda(), x["w_uv"].cuda(), k_c, v, None)
    got = []
    for value in (0.0, fill):
        cache, k, vv = zero.clone(), k_c.clone(), v.clone()
        for plane in (cache, k, vv):
            plane[free] = value
        got.append((*_absorb(bd, w, q_hat, cache, table, page, sl, S, status),
                    *_gqa(bd, w, q, k, vv, cache[:, w.r_kv:], table, page, sl, S, status)))
    assert int(status.item()) == 0
    for a, b, what in zip(*got, ("absorb o", "absorb lse", "gqa o", "gqa lse")):
        assert not torch.isnan(b).any(), what
        assert torch.equal(a, b), what


@pytest.mark.parametrize("dims", [CANON, LLAMA, dict(LLAMA, h_q=16)])
@pytest.mark.parametrize("page,S,s_q", [(16, 1, 1), (32, -3, 2), (64, 1, 2), (64, 3, 1), (192, -2, 1), (128, 2, 1)])
def test_probabilities_keep_their_24_bits(dims, page, S, s_q):
    """Value rows are unit vectors, so every output element is one probability, and the keys are too, so every score is one
    query element, exactly.  What is left are the roundings of x = s log2(e) (|s| <= 1/2: 3 * 2^-25), ex2 (2^-22) in the
    probability and in the sum, and a few of 2^-24 in the normalisation and the merge: below 2^-20 in all.  Probabilities cut to
    16 bits miss by up to 2^-17."""
    seqlens = np.array([1, 2, 5, 16, 63, 64, 65, 100, 127, 128], dtype=np.int32)
    w = synth.Workload("onehot", batch=len(seqlens), s_q=s_q, dtype="bf16", seed=303, **dims)
    gen = torch.Generator().manual_seed(304)
    scale = 0.25
    rows = torch.cat([torch.eye(128)[:n] for n in seqlens]).bfloat16()
    starts = np.concatenate([[0], np.cumsum(seqlens)[:-1]])
    pool, table = synth.to_paged(rows, starts, seqlens, page, seed=305, fill=0.0)
    pool, table, sl = pool.cuda(), table.cuda(), torch.from_numpy(seqlens).cuda()
    cache = torch.zeros((pool.shape[0], w.r_kv + w.d_r), dtype=torch.bfloat16, device="cuda")
    cache[:, :128] = pool
    k_c = pool[:, None, :].expand(-1, w.g, -1).contiguous()
    x = (4 * torch.rand((w.batch, s_q, w.h_q, 128), generator=gen) - 2).bfloat16()
    zeros = torch.zeros((w.batch, s_q, w.h_q, w.r_kv - 128 + w.d_r), dtype=torch.bfloat16)
    q_hat, q = torch.cat([x, zeros], -1).cuda(), torch.cat([x, zeros[..., :w.d_r]], -1).cuda()
    bd = B.make_dims(w.h_q, w.g, w.d_h, w.r_kv, w.d_r)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s = scale * x.double()
    for b, n in enumerate(seqlens):
        for p in range(s_q):
            s[b, p, :, max(0, int(n) - (s_q - 1 - p)):] = -np.inf
    ref = torch.nan_to_num(torch.softmax(s, -1))  # a query that sees nothing gives 0
    for o, lse, what in ((*_absorb(bd, w, q_hat, cache, table, page, sl, S, status, scale), "absorb"),
                         (*_gqa(bd, w, q, k_c, k_c, cache[:, w.r_kv:], table, page, sl, S, status, scale), "gqa")):
        out = torch.empty((w.batch, s_q, w.h_q, o.shape[-1]), device="cuda")
        B.gqla_combine_splits(o, lse, out)
        got = out.double().cpu()
        assert int(status.item()) == 0 and not got[..., 128:].any()
        err = ((got[..., :128] - ref).abs() / torch.where(ref > 0, ref, torch.ones(()).double())).max()
        assert err <= 2.0 ** -20, (what, float(err))


@pytest.mark.parametrize("h_q,s_q", [(128, 1), (128, 2), (32, 1)])
@pytest.mark.parametrize("page,S", [(16, 1), (64, -2), (128, 2)])
def test_infinite_values_stay_infinite_on_the_gqa_path(h_q, s_q, page, S):
    """An infinity among the values of a sequence reaches the output as itself (it is a sum with positive weights), also where the
    second and third term of a probability are zero or negative; the sequences beside it are untouched."""
    seqlens = np.array([2, 40, 70, 200], dtype=np.int32)
    w = synth.Workload("inf", batch=len(seqlens), s_q=s_q, dtype="bf16", seed=308, **dict(CANON, h_q=h_q))
    x = synth.make_inputs(w, seqlens=seqlens)
    table = synth.to_paged(x["cache"], x["seq_start"], seqlens, page, seed=309)[1].cuda()
    n = 1 + int(table.max()) + 3
    gen = torch.Generator().manual_seed(310)
    k_c, v = (torch.randn((n * page, w.g, w.d_h), generator=gen).bfloat16().cuda() for _ in range(2))
    k_r = torch.randn((n * page, w.d_r), generator=gen).bfloat16().cuda()
    q = torch.cat([x["q_c"], x["q_r"]], -1).contiguous()
    q[0] = 0  # equal probabilities: their further terms are zero
    bd = B.make_dims(w.h_q, w.g, w.d_h, w.r_kv, w.d_r)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def step():
        o, lse = _gqa(bd, w, q.cuda(), k_c, v, k_r, table, page, x["seqlens"].cuda(), S, status)
        out = torch.empty((w.batch, s_q, w.h_q, w.d_h), device="cuda")
        B.gqla_combine_splits(o, lse, out)
        return out

    ref = step()
    for b in (0, 2):
        row = int(table[b, 0]) * page  # the sequence's first row, which every query sees
        v[row, :, :3], v[row, :, 3:7] = np.inf, -np.inf
        ref[b, ..., :3], ref[b, ..., 3:7] = np.inf, -np.inf
    assert torch.equal(step(), ref) and int(status.item()) == 0


@pytest.mark.parametrize("dims", [CANON, LLAMA, dict(CANON, h_q=64), dict(CANON, h_q=28, g=4), dict(LLAMA, h_q=16)])
@pytest.mark.parametrize("page,S,s_q,tensor_cores", [
    (16, 1, 1, True), (16, -9, 2, True), (32, -3, 1, True), (48, 5, 2, True), (64, 1, 2, True), (64, -7, 1, True), (192, -3, 2, True),
    (128, 3, 1, True), (256, 6, 2, True), (128, -3, 1, True), (64, 2, 3, True), (24, 1, 1, False), (8, -3, 2, False)])
def test_which_kernels_serve_a_page_size(dims, page, S, s_q, tensor_cores):
    """The generic kernels give the same bits under either policy; the tensor-core kernels sum in another order and do not.
    GQA calls over small pages leave the tensor cores beyond 32 padded query rows per group."""
    seqlens = np.array([700, 129, 333], dtype=np.int32)
    w = synth.Workload("route", batch=len(seqlens), s_q=s_q, dtype="bf16", seed=311, **dims)
    x = synth.make_inputs(w, seqlens=seqlens, q_gain=2.0)
    pool, table = synth.to_paged(x["cache"], x["seq_start"], seqlens, page, seed=312)
    pool, table, sl = pool.cuda(), table.cuda(), x["seqlens"].cuda()
    bd = B.make_dims(w.h_q, w.g, w.d_h, w.r_kv, w.d_r)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    q = torch.cat([x["q_c"], x["q_r"]], -1).contiguous().cuda()
    q_hat = torch.empty((w.batch, s_q, w.h_q, w.d_abs), dtype=torch.bfloat16, device="cuda")
    k_c, v = (torch.empty((pool.shape[0], w.g, w.d_h), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    B.gqla_absorb_q(bd, x["q_c"].cuda(), x["q_r"].cuda(), x["w_uk"].cuda(), q_hat)
    B.gqla_expand_cache(bd, pool, x["w_uk"].cuda(), x["w_uv"].cuda(), k_c, v, None)
    runs = []
    for policy in (B.POLICY_AUTO, B.POLICY_GENERIC):
        B.set_policy(policy)
        try:
            runs.append((_absorb(bd, w, q_hat, pool, table, page, sl, S, status)[0],
                         _gqa(bd, w, q, k_c, v, pool[:, w.r_kv:], table, page, sl, S, status)[0]))
        finally:
            B.set_policy(B.POLICY_AUTO)
    assert int(status.item()) == 0
    rows = (1 << (w.h_q // w.g - 1).bit_length()) * (1 << (s_q - 1).bit_length())
    small = page % 128 != 0 or S > 1
    assert torch.equal(runs[0][0], runs[1][0]) == (not tensor_cores)
    assert torch.equal(runs[0][1], runs[1][1]) == (not tensor_cores or (small and rows > 32))
