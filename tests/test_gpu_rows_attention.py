"""Attention of the (K + 1)-row pass: the edges of its chunks of 16 keys and its iterations of 14 (nine rows: 12) of them, for every number of
rows, on both sides of the line between its two builds; keys and values that overflowed the cache; small products; the same result
however cycles are called (run on a B200)."""
import numpy as np
import pytest
import torch

import paper_2604_14612_b200 as cl
from test_gpu_wide_attention import _model

pytestmark = pytest.mark.gpu

DT = {"bf16": torch.bfloat16, "fp16": torch.float16}
V = 256


def _random_model(wd, heads, kv_heads, hd):
    d, kvd, F = heads * hd, kv_heads * hd, 128
    g = torch.Generator(device="cuda").manual_seed(heads * hd)
    t = lambda r, c, s=0.05: (torch.randn((r, c), generator=g, device="cuda") * s).to(DT[wd])
    o = lambda: torch.ones(d, device="cuda")
    return d, F, dict(embed=t(V, d, 1.0), lm_head=t(V, d), final_norm=o(), wq=[t(d, d)], wk=[t(kvd, d)], wv=[t(kvd, d)], wo=[t(d, d)],
                      wg=[t(F, d)], wu=[t(F, d)], wd=[t(d, F)], norm1=[o()], norm2=[o()])


@pytest.mark.parametrize("wd,heads,kv_heads,hd", [("bf16", 2, 2, 64), ("fp16", 4, 2, 128), ("bf16", 40, 40, 64), ("fp16", 37, 37, 64), ("bf16", 8, 1, 128)])
def test_every_number_of_rows_and_cached_keys(monkeypatch, wd, heads, kv_heads, hd):
    """Against the CUDA-core pass, on the same cache.  Heads in 8, 8, 3, 4 and 8 parts.  Both passes round the new values to the storage
    type; an operand of 16 bits (2^-17 off) decides about one bf16 value in 2^8 the other way, by 2^-9: 2^-9 * 2^-4 = 1.2e-4 of the
    output where one key is all there is, four times that as bound."""
    d, F, W = _random_model(wd, heads, kv_heads, hd)
    out = {}
    for off in ("0", "1"):
        monkeypatch.setenv("CL_DISABLE_ROWS_KERNEL", off)
        ctx = cl.Context(1, d, heads, F, V, 2000, wd, 1e-5, 1e4, tap_positions=16, n_kv_heads=kv_heads)
        ctx.cl_load(W)
        res = []
        # around the lines between the two builds (8 parts: 8 rows 256, 9 384, 5 to 7 512, 4 768, 3 1024); last parts of 192 and 193 keys, whole
        # iterations of nine rows, behind which the pass's own chunk stands alone (8 parts 1536, 3 576, 4 768)
        for n in (17, 18, 31, 33, 127, 129, 256, 257, 273, 384, 385, 401, 447, 448, 449, 512, 513, 529, 576, 579, 768, 769, 772, 895, 897,
                  1024, 1025, 1536, 1544, 1791, 1900):
            ctx.cl_prefill((np.arange(n) * 7 + n).astype(np.int32) % V)
            for T in range(1, 10):
                ctx.cl_rollback(n, n % V)
                ctx.cl_force_tokens((np.arange(T - 1) * 3 + 1).astype(np.int32))
                res.append((n, T, ctx.cl_verify(T, tap_hidden=True, want_logits=True)["logits"].copy()))
        for n in (1, 2, 8):                     # short prompts: chunks of rows behind nothing
            ctx.cl_prefill((np.arange(n) * 5 + 2).astype(np.int32) % V)
            ctx.cl_rollback(n, 3)
            ctx.cl_force_tokens([4, 5])
            res.append((n, 3, ctx.cl_verify(3, want_logits=True)["logits"].copy()))
        out[off] = res
        ctx.close()
    for (n, T, x), (_, _, y) in zip(out["0"], out["1"]):
        rel = np.linalg.norm(x - y) / np.linalg.norm(y)
        assert rel <= 5e-4, (n, T, rel)


@pytest.mark.parametrize("n", [600, 40])   # (many keys a part and few: each build)
@pytest.mark.parametrize("T", [1, 5, 9])
def test_keys_that_score_minus_infinity_have_no_weight(T, n):
    """fp16 keys of 1e5 are infinite; against a negative query they score -inf, so the first token's value is the whole output."""
    g = torch.Generator().manual_seed(6)
    values, first = (1.0 + torch.rand(256, generator=g)) * 500, 1.0 + torch.rand(256, generator=g)
    first[:3] = 0.0
    ctx, emb, _ = _model("fp16", 4, n + 8, [-32.0, -1.0, -3.3, -0.01], values, first_key=0.0, other_key=1e5, first_value=first)
    ctx.cl_prefill(np.concatenate([[0], 1 + np.arange(n - 1) % 1000]).astype(np.int32))
    ctx.cl_rollback(n, 7)
    ctx.cl_force_tokens(np.arange(1, T).astype(np.int32))
    ctx.cl_verify(T, tap_hidden=True)
    ring = ctx.cl_read_hidden_ring().double().numpy()[0]
    ctx.close()
    got = ring[[(n + t) % 512 for t in range(T)]]
    want = (first / 16.0).half().double().numpy() * 16.0
    assert np.isfinite(got).all()
    assert np.abs(got - emb[[7] + list(range(1, T))] - want)[:, 3:].max() <= 2e-3          # half a step of fp16 at 2 is 1e-3


@pytest.mark.parametrize("n", [600, 100])
@pytest.mark.parametrize("T", [1, 5, 9])
def test_a_key_with_weight_behind_keys_that_score_minus_infinity(T, n):
    """All cached keys score -inf; the pass's first token, the first to score 0, is the whole output of every row."""
    g = torch.Generator().manual_seed(6)
    values, first = (1.0 + torch.rand(256, generator=g)) * 500, 1.0 + torch.rand(256, generator=g)
    first[:3] = 0.0
    ctx, emb, _ = _model("fp16", 4, n + 16, [-32.0, -1.0, -3.3, -0.01], values, first_key=0.0, other_key=1e5, first_value=first)
    ctx.cl_prefill((1 + np.arange(n) % 1000).astype(np.int32))
    ctx.cl_rollback(n, 0)
    ctx.cl_force_tokens(np.arange(1, T).astype(np.int32))
    ctx.cl_verify(T, tap_hidden=True)
    ring = ctx.cl_read_hidden_ring().double().numpy()[0]
    ctx.close()
    got = ring[[(n + t) % 512 for t in range(T)]]
    want = (first / 16.0).half().double().numpy() * 16.0
    assert np.isfinite(got).all()
    assert np.abs(got - emb[[0] + list(range(1, T))] - want)[:, 3:].max() <= 2e-3          # half a step of fp16 at 2 is 1e-3


@pytest.mark.parametrize("n", [40, 600])   # (each build: keys walked, tensor cores)
@pytest.mark.parametrize("T", [5, 9])
def test_a_candidate_whose_value_overflows_leaves_the_rows_before_it_alone(T, n):
    """Token 0 has values of 1e5, infinite in fp16: rows that do not attend to it are the same to the bit, rows that do are not finite."""
    ctx, _, _ = _model("fp16", 4, n + 16, [1.0, 2.0, -1.0, 0.5], torch.ones(256), first_value=1e5)
    rows = {}
    for third in (0, 5):
        ctx.cl_prefill((1 + np.arange(n)).astype(np.int32))
        ctx.cl_rollback(n, 7)
        ctx.cl_force_tokens(np.array([1, 2, third] + list(range(10, 6 + T)), np.int32))
        ctx.cl_verify(T, tap_hidden=True)
        rows[third] = ctx.cl_read_hidden_ring().double().numpy()[0][[(n + t) % 512 for t in range(T)]]
    ctx.close()
    assert np.isfinite(rows[5]).all()
    assert np.array_equal(rows[0][:3], rows[5][:3])
    assert not np.isfinite(rows[0][3:, 3:]).any()


@pytest.mark.parametrize("value", [500.0, 1e5])
@pytest.mark.parametrize("n", [40, 600])
@pytest.mark.parametrize("T", [5, 9])
def test_a_candidate_whose_key_overflows_has_no_weight_against_negative_queries(T, n, value):
    """Token 0 has keys of 1e5, infinite in fp16, that score -inf, and values that may be infinite too; all others score 0 and have the same
    value: the output of every row."""
    g = torch.Generator().manual_seed(7)
    values = 1.0 + torch.rand(256, generator=g)
    values[:3] = 0.0
    ctx, emb, v = _model("fp16", 4, n + 16, [-32.0, -1.0, -3.3, -0.01], values, first_key=1e5, first_value=value)
    ctx.cl_prefill((1 + np.arange(n)).astype(np.int32))
    ctx.cl_rollback(n, 7)
    tokens = [7, 1, 2, 0] + list(range(10, 6 + T))
    ctx.cl_force_tokens(np.array(tokens[1:], np.int32))
    ctx.cl_verify(T, tap_hidden=True)
    got = ctx.cl_read_hidden_ring().double().numpy()[0][[(n + t) % 512 for t in range(T)]]
    ctx.close()
    assert np.isfinite(got).all()
    assert np.abs(got - emb[tokens] - v)[:, 3:].max() <= 2e-3          # half a step of fp16 at 2 is 1e-3


@pytest.mark.parametrize("wd", ["bf16", "fp16"])
@pytest.mark.parametrize("T,n", [(3, 1100), (5, 600), (9, 600), (5, 40)])
def test_small_products_beside_a_large_one_are_not_cut_off(wd, T, n):
    """Two kinds of keys score 1024 and 1024 + 2.25 * 2^-13; the excess is three products of 0.75 * 2^-13, each in another instruction of
    the score's contraction.  Products, scores and the scaling by 1/8 are exact (marks are 16 after the norm, numbers have two bits), so
    a score is off by roundings alone: one step of 2^-13, where an accumulator that cuts off would lose all three products.  The rows of
    the pass themselves have keys of 0 (no weight); values are u and -u, so the hidden state is -u tanh(excess / 2)."""
    heads, d, steps = 4, 256, 2.0 ** -13
    g = torch.Generator().manual_seed(11)
    emb = (torch.rand((V, d), generator=g) - 0.5) * 1e-3
    emb[:, :6] = 0.0
    emb[:, :3] = 256.0
    for i in range(V):
        emb[i, 3 + min(i // 100, 2)] = 256.0   # tokens 0 .. 99, 100 .. 199, from 200 on; four columns of 256 among 256: normalised 8, gain 2
    emb = emb.to(DT[wd])
    z = lambda r, c: torch.zeros((r, c), dtype=torch.float32)
    wq, wk, wv = z(d, d), z(d, d), z(d, d)
    u = (1.0 + torch.rand(d, generator=g)).to(DT[wd]).float()
    for h in range(heads):
        # (dimensions 16 .. 31 and their partners 48 .. 63 rotate by less than 1e-6 over all positions; none of these is another's partner)
        for e, q, k in ((16, 64.0, 128.0), (20, 2.0 ** -5, 0.75 * 2.0 ** -5), (56, 2.0 ** -5, 0.75 * 2.0 ** -5), (60, 2.0 ** -5, 0.75 * 2.0 ** -5)):
            wq[64 * h + e, 0] = q / 16.0
            wk[64 * h + e, 4] = k / 16.0
            if e == 16:
                wk[64 * h + e, 3] = k / 16.0
    wv[:, 3], wv[:, 4] = u / 16.0, -u / 16.0
    wv[:6] = 0.0
    t = lambda x: x.to(DT[wd]).cuda()
    ctx = cl.Context(1, d, heads, 64, V, n + 16, wd, 1e-5, 1e20, tap_positions=512)
    ctx.cl_load(dict(embed=emb.cuda(), lm_head=t(z(V, d)), final_norm=torch.ones(d).cuda(), wq=[t(wq)], wk=[t(wk)], wv=[t(wv)], wo=[t(torch.eye(d))],
                     wg=[t(z(64, d))], wu=[t(z(64, d))], wd=[t(z(d, 64))], norm1=[torch.full((d,), 2.0).cuda()], norm2=[torch.ones(d).cuda()]))
    ctx.cl_prefill((np.arange(n) % 2 * 100 + np.arange(n) // 2 % 100).astype(np.int32))
    rows = 200 + np.arange(T)
    ctx.cl_rollback(n, int(rows[0]))
    ctx.cl_force_tokens(rows[1:].astype(np.int32))
    ctx.cl_verify(T, tap_hidden=True)
    ring = ctx.cl_read_hidden_ring().double().numpy()[0]
    ctx.close()
    att = ring[[(n + i) % 512 for i in range(T)]] - emb.double().numpy()[rows]
    excess = -2.0 * np.arctanh((att / u.double().numpy())[:, 6:].mean(1))
    assert np.abs(excess / steps - 2.25).max() <= 1.0, excess / steps


@pytest.mark.parametrize("K,n,gen", [(8, 250, 160), (4, 300, 240)])
def test_single_cycles_and_one_call_and_several_compute_the_same(K, n, gen):
    """Generation across the lines between the two builds of the pass (heads in 8 parts: 384 cached keys with nine rows, 512 with five):
    which one a position takes does not depend on how the cycles are called, so tokens and the logits behind them agree to the bit.
    (Calls end where a cycle ends: a cycle that begins elsewhere splits the keys differently.)"""
    d, F, W = _random_model("bf16", 4, 4, 64)
    W = {k: v * 2 if isinstance(v, list) else v for k, v in W.items()}   # (two layers: the second one's keys depend on the attention)
    ctx = cl.Context(2, d, 4, F, V, n + gen + 64, "bf16", 1e-5, 1e4, tap_positions=16, n_kv_heads=4)
    ctx.cl_load(W)
    prompt = (np.arange(n) * 7 + n).astype(np.int32) % V

    def logits_behind(toks):
        ctx.cl_force_tokens([4, 5])
        return toks, ctx.cl_verify(3, want_logits=True)["logits"].copy()

    ctx.cl_prefill(prompt)
    toks, ends = [], [0]
    while len(toks) < gen:
        ctx.cl_draft(K)
        ctx.cl_verify(K + 1)
        toks += [int(x) for x in ctx.cl_accept()[1]]
        ends.append(len(toks))
    out = [logits_behind(toks)]
    for cuts in (ends[::len(ends) - 1], [ends[0], ends[len(ends) // 3], ends[2 * len(ends) // 3], ends[-1]]):
        ctx.cl_prefill(prompt)
        toks = []
        for a, b in zip(cuts, cuts[1:]):
            toks += [int(x) for x in ctx.cl_generate(K, b - a)[0]]
        out.append(logits_behind(toks))
    ctx.close()
    for toks, logits in out[1:]:
        assert toks == out[0][0]
        assert np.array_equal(logits, out[0][1])
