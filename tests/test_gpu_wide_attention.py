"""Accuracy of the prompt pass's attention against the exact result (run on a B200).

A one-layer model whose attention output can be written down: every token but the first has the same query, key and value,
the first token's key scores `gap` above theirs in each head and its value is zero, the output projection is the identity and
the FFN is zero.  The hidden state of row t is then its embedding plus, per head,

    n p v / (1 + n p),   n = t keys of weight p = exp(-gap)

Keys, values and queries are exact in the storage type; hidden states come back in it, and embeddings carry a known offset of
about one of its steps, so that its rounding averages out over rows and columns.
"""
import numpy as np
import pytest
import torch

import paper_2604_14612_b200 as cl

pytestmark = pytest.mark.gpu

DT = {"bf16": torch.bfloat16, "fp16": torch.float16}
V, P = 1024, 512


def _model(wd, heads, n, gaps, values, first_key=16.0, other_key=0.0, first_value=0.0):
    """(context, embedding, values [d]): d = 64 heads; queries and keys live in dimension 31 of a head, which rotates by
    less than 1e-18 per position; the normalised first token is 16 in column 0, the others 16 in column 1 (both in column 2)."""
    d = 64 * heads
    g = torch.Generator().manual_seed(n)
    big = 256.0
    emb = (torch.rand((V, d), generator=g) - 0.5) * (2e-3 if wd == "fp16" else 1.6e-2)
    emb[:, :3] = 0.0
    emb[0] = 0.0
    emb[0, [0, 2]] = big                       # two columns of 256: their normalised value is sqrt(d / 2) times the gain
    emb[1:, 1] = big
    emb[1:, 2] = big
    emb = emb.to(DT[wd])
    gain = torch.full((d,), float(16.0 * np.sqrt(2.0 / d)), dtype=torch.float32)
    z = lambda r, c: torch.zeros((r, c), dtype=torch.float32)
    wq, wk, wv, wo = z(d, d), z(d, d), z(d, d), torch.eye(d)
    for h, gap in enumerate(gaps):
        wq[64 * h + 31, 2] = gap / 32.0        # q = gap / 2, k = 16: the score of the first key is q k / 8 = gap
        wk[64 * h + 31, 0] = first_key / 16.0
        wk[64 * h + 31, 1] = other_key / 16.0
    wv[:, 1] = values / 16.0
    wv[:, 0] = first_value / 16.0
    wv[:3] = 0.0
    t = lambda x: x.to(DT[wd]).cuda()
    w = dict(embed=emb.cuda(), lm_head=t(z(V, d)), final_norm=torch.ones(d).cuda(), wq=[t(wq)], wk=[t(wk)], wv=[t(wv)], wo=[t(wo)],
             wg=[t(z(64, d))], wu=[t(z(64, d))], wd=[t(z(d, 64))], norm1=[gain.cuda()], norm2=[torch.ones(d).cuda()])
    ctx = cl.Context(1, d, heads, 64, V, n + 8, wd, 1e-5, 1e20, tap_positions=P)
    ctx.cl_load(w)
    return ctx, emb.double().numpy(), t(wv[:, 1] * 16.0).double().cpu().numpy()


def _hidden(ctx, n, tokens):
    """Rows n - P .. n - 1 after the layer, fp64."""
    ctx.cl_prefill(tokens, tap_hidden=True)
    ring = ctx.cl_read_hidden_ring().double().numpy()[0]
    return ring[[t % P for t in range(n - P, n)]]


@pytest.mark.parametrize("wd", ["fp16", "bf16"])
def test_light_keys_under_a_heavy_one_keep_their_weight(wd):
    """4095 keys under one that scores up to 20 more and has no value: together they carry down to 0.0008 % of the mass and all
    of the output, so it is as exact as their weights and the sums of them.  Largest error: half a step of the storage type.
    Mean over 512 rows of 64 columns: the rounding leaves 2^-10 / sqrt(12 * 32768) of the value in fp16 (four times that:
    6.2e-6), a score of 20 with a relative error of 2^-23 another 2.4e-6, weights and sums 1e-6; bf16 has eight times the step
    and a query of 16 bits (score error 20 * 2^-17 / sqrt(12))."""
    n, gaps = 4096, [0.5, 10.0, 17.5, 20.0]
    g = torch.Generator().manual_seed(5)
    scale = torch.tensor([1.0, 8.0, 8192.0, 16384.0]).repeat_interleave(64)
    values = ((1.0 + torch.rand(256, generator=g)) * scale).to(DT[wd]).float()
    values[:3] = 0.0
    ctx, emb, v = _model(wd, 4, n, gaps, values)
    tokens = np.concatenate([[0], 1 + np.arange(n - 1) % (V - 1)]).astype(np.int32)
    got = _hidden(ctx, n, tokens)
    ctx.close()
    t = np.arange(n - P, n, dtype=np.float64)[:, None]
    p = np.exp(-np.repeat(np.array(gaps), 64))[None]
    att = t * p * v[None] / (1 + t * p)
    err = (got - emb[tokens[n - P:]] - att)[:, 3:] / att[:, 3:]
    head = np.arange(3, 256) // 64
    for h in range(4):
        e = err[:, head == h]
        assert np.abs(e).max() <= (2e-3 if wd == "fp16" else 1.6e-2), (gaps[h], np.abs(e).max())
        assert abs(e.mean()) <= (1e-5 if wd == "fp16" else 1e-4), (gaps[h], e.mean())


def test_keys_that_overflowed_the_cache_and_score_minus_infinity_have_no_weight():
    """Keys of 1e5 are infinite in an fp16 cache.  Against a negative query they score -inf: their weight is 0 and the first
    token's value is the whole output of every row."""
    n = 600
    g = torch.Generator().manual_seed(6)
    values, first = (1.0 + torch.rand(256, generator=g)) * 500, 1.0 + torch.rand(256, generator=g)
    first[:3] = 0.0
    ctx, emb, _ = _model("fp16", 4, n, [-32.0, -1.0, -3.3, -0.01], values, first_key=0.0, other_key=1e5, first_value=first)
    tokens = np.concatenate([[0], 1 + np.arange(n - 1) % (V - 1)]).astype(np.int32)
    got = _hidden(ctx, n, tokens)
    ctx.close()
    want = (first / 16.0).half().double().numpy() * 16.0
    assert np.isfinite(got).all()
    assert np.abs(got - emb[tokens[n - P:]] - want)[:, 3:].max() <= 2e-3          # half a step of fp16 at 2 is 1e-3


@pytest.mark.parametrize("wd,steps", [("fp16", [0.5, 1.0, 0.5, 0.0]), ("bf16", [0.5, 1.0, 4.0, 0.0])])
def test_large_scores_whose_maximum_rises_from_tile_to_tile(wd, steps):
    """Eight tiles of 64 keys, a score each, then keys without weight.  Scores are exact (the normalised marks are 16, keys and
    queries have few bits), from 100, 246 and 992 on in steps that the storage type holds; in the last head all are 9.4e7.  Values have alternating signs and
    cancel up to their own rounding, so that hidden states stay near 1e-3 and their rounding, averaged over rows and columns, near 1e-8.
    Bound, of the values: a weight is off by 2^-22 at most (two steps of expf), by 2^-24 for each of eight rescalings and two
    cut-off sums; with signs at random 4 * 2^-24 * sqrt(2^2 + 8 + 2) = 8.9e-7."""
    heads, d, n = 4, 256, 1024
    g = torch.Generator().manual_seed(9)
    starts, queries = [100.0, 246.0, 992.0, 32768.0], [8.0, 8.0, 8.0, 16.0 * 1440.0]
    emb = (torch.rand((V, d), generator=g) - 0.5) * 1e-3
    emb[:, :16] = 0.0
    emb[:, :3] = 256.0
    tokens = np.concatenate([np.repeat(np.arange(8), 64), np.full(n - 512, 8)]) * 100
    tokens = (tokens + np.arange(n) % 64).astype(np.int32)
    for i in range(V):
        emb[i, 3 + min(i // 100, 8)] = 256.0   # four columns of 256 among 256: normalised 8, with the gain 16
    emb = emb.to(DT[wd])
    z = lambda r, c: torch.zeros((r, c), dtype=torch.float32)
    wq, wk, wv, wo = z(d, d), z(d, d), z(d, d), torch.eye(d)
    u = 1.0 + torch.rand(64, generator=g)
    weight = np.zeros((heads, 8))
    for h in range(heads):
        score = (starts[h] + steps[h] * np.arange(8)) * queries[h] / 8.0
        weight[h] = np.exp(score - score.max())
        wq[64 * h + 31, 0] = queries[h] / 16.0
        sign = np.array([1.0, -1.0] * 4)
        sign[7] = -(weight[h] * sign)[:7].sum()
        for j in range(8):
            wk[64 * h + 31, 3 + j] = (starts[h] + steps[h] * j) / 16.0
            wv[64 * h : 64 * h + 64, 3 + j] = u * float(sign[j]) / 16.0
    wv[:16] = 0.0
    t = lambda x: x.to(DT[wd]).cuda()
    ctx = cl.Context(1, d, heads, 64, V, n + 8, wd, 1e-5, 1e20, tap_positions=P)
    ctx.cl_load(dict(embed=emb.cuda(), lm_head=t(z(V, d)), final_norm=torch.ones(d).cuda(), wq=[t(wq)], wk=[t(wk)], wv=[t(wv)], wo=[t(wo)],
                     wg=[t(z(64, d))], wu=[t(z(64, d))], wd=[t(z(d, 64))], norm1=[torch.full((d,), 2.0).cuda()], norm2=[torch.ones(d).cuda()]))
    got = _hidden(ctx, n, tokens) - emb.double().numpy()[tokens[n - P:]]
    ctx.close()
    value = (t(wv)[:, 3:11] * 16.0).double().cpu().numpy().reshape(heads, 64, 8)
    want = (value * weight[:, None]).sum(2) / weight.sum(1)[:, None]
    err = ((got.reshape(P, heads, 64) - want) / u.double().numpy()).mean(0)
    for h in range(heads):
        e = err[h, 16 if h == 0 else 0:].mean()
        assert abs(e) <= 8.9e-7, (starts[h], e)
