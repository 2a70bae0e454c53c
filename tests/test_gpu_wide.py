"""The wide prompt pass at the edges of its tiles (run on a B200).

Operand rows come in tiles of 256, a rest of at most 128 rows as a half tile; the attention walks 64 rows by 64 keys; a
matrix whose width is no multiple of 64 ends in a partial K block.  Every length is compared with the 8-row passes over the
same prompt, which share none of these kernels.
"""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2604_14612_b200 as cl
import synth

pytestmark = pytest.mark.gpu

SHAPES = {
    "hd64": dict(d_model=768, n_heads=12, d_ffn=2048),
    "hd128_grouped_ragged_ffn": dict(d_model=512, n_heads=4, n_kv_heads=2, d_ffn=712),
}


@pytest.mark.parametrize("shape,wd,n", [("hd64", "bf16", 64), ("hd64", "bf16", 128), ("hd64", "fp16", 129), ("hd64", "bf16", 256),
                                        ("hd64", "bf16", 257), ("hd64", "fp16", 384), ("hd64", "bf16", 385), ("hd64", "bf16", 512),
                                        ("hd128_grouped_ragged_ffn", "bf16", 33), ("hd128_grouped_ragged_ffn", "fp16", 65),
                                        ("hd128_grouped_ragged_ffn", "bf16", 300), ("hd128_grouped_ragged_ffn", "fp16", 1025)])
def test_wide_pass_at_tile_edges(monkeypatch, shape, wd, n):
    """First token, hidden taps and the logits of a pass that reads the whole cache.  Both sides keep 16 mantissa bits of the
    activations and the same cache rounding: taps agree to one bf16 ulp at the top of their range, logits to half of the
    1e-2 that a model of this depth is allowed against the oracle."""
    sh = dataclasses.replace(synth.WORKLOADS["C2"].shape, n_layers=2, max_seq=n + 16, weight_dtype=wd, vocab=4000,
                             **{"n_kv_heads": 0, **SHAPES[shape]})
    W = synth.make_weights(sh, 21, device="cuda")
    prompt = synth.make_prompt(21, n, sh.vocab)
    out = {}
    for wide in (0, 1):
        monkeypatch.setenv("CL_DISABLE_WIDE_PREFILL", "0" if wide else "1")
        ctx = cl.Context.from_shape(sh, tap_positions=16)
        ctx.cl_load(W)
        first = ctx.cl_prefill(prompt, tap_hidden=True)
        ring = ctx.cl_read_hidden_ring().float().numpy()
        ctx.cl_rollback(n, 7)
        ctx.cl_force_tokens([11, 22])
        out[wide] = (first, ring, ctx.cl_verify(3, want_logits=True)["logits"].copy())
        ctx.close()
    scale = max(1.0, float(np.abs(out[0][1]).max()))
    assert np.abs(out[0][1] - out[1][1]).max() <= 2 ** -7 * scale
    assert np.abs(out[0][2] - out[1][2]).max() <= 5e-3
    ctx = cl.Context.from_shape(sh)
    ctx.cl_load(W)
    ctx.cl_prefill(prompt[:-1])
    ctx.cl_rollback(n - 1, int(prompt[-1]))
    lg = ctx.cl_verify(1, want_logits=True)["logits"][0]
    assert lg[out[0][0]] - lg[out[1][0]] < 1e-2 and lg.max() - lg[out[1][0]] < 1e-2   # the same token up to a near tie


def test_wide_attention_takes_any_score_range():
    """Queries large enough to overflow fp16 parts if they were not scaled: the pass stays finite and follows the 8-row one."""
    sh = dataclasses.replace(synth.WORKLOADS["C2"].shape, n_layers=1, max_seq=96, weight_dtype="fp16", vocab=1024)
    W = synth.make_weights(sh, 22, device="cuda")
    W["wq"][0] = (W["wq"][0].float() * 3e4).to(torch.float16)             # queries of about 1e4 .. 1e5, |scores| up to 1e5
    prompt = synth.make_prompt(22, 80, sh.vocab)
    got = []
    for wide in (0, 1):
        with pytest.MonkeyPatch.context() as mp:
            mp.setenv("CL_DISABLE_WIDE_PREFILL", "0" if wide else "1")
            ctx = cl.Context.from_shape(sh, tap_positions=32)
            ctx.cl_load(W)
            ctx.cl_prefill(prompt, tap_hidden=True)
            got.append(ctx.cl_read_hidden_ring().float().numpy())
            ctx.close()
    assert np.isfinite(got[1]).all()
    # scores of 1e5 with a relative error of 2^-16 (the normalised rows' hi / lo parts) move a weight only where two keys
    # tie to within a unit: rows with one dominant key agree, so all but a few do
    row = np.abs(got[0] - got[1]).max(axis=2) <= 2 ** -7 * max(1.0, float(np.abs(got[0]).max()))
    assert row.mean() >= 0.9


@pytest.mark.parametrize("wd,n", [("fp16", 512), ("fp16", 300), ("bf16", 256)])
def test_products_of_full_tiles_against_fp64(wd, n):
    """The FFN half of a layer of width 4096 (sums over 4096 and 11008 elements: several accumulation chains per tile, shares that
    end inside a tile), every row against fp64.  Each hidden value is the exact one rounded to the storage type, up to what the
    sums lose: the accumulator of the tensor core cuts off, which makes results smaller, about 2^-26 of them per instruction of a
    chain of 64 (8 K blocks, hi and lo parts): 1e-6 per matrix, three matrices and the slope of SiLU: 4e-6.  Seen through the
    storage type's rounding, 2^-11 / sqrt(3) of a value (fp16) over n * 4096 values, 3e-7 (bf16: eight times that)."""
    d, F, dt = 4096, 11008, {"fp16": torch.float16, "bf16": torch.bfloat16}[wd]
    g = torch.Generator(device="cuda").manual_seed(n)
    rnd = lambda r, c, std: (torch.randn((r, c), generator=g, device="cuda") * std).to(dt)
    zero = torch.zeros((d, d), device="cuda", dtype=dt)
    V = 2000
    W = dict(embed=rnd(V, d, 0.5), lm_head=rnd(V, d, 0.02), final_norm=torch.ones(d, device="cuda"), wq=[zero], wk=[zero], wv=[zero], wo=[zero],
             wg=[rnd(F, d, 0.02)], wu=[rnd(F, d, 0.02)], wd=[rnd(d, F, 0.02)], norm1=[torch.ones(d, device="cuda")],
             norm2=[1.0 + 0.1 * torch.randn(d, generator=g, device="cuda")])
    ctx = cl.Context(1, d, 32, F, V, n + 8, wd, tap_positions=n)
    ctx.cl_load(W)
    prompt = synth.make_prompt(23, n, V)
    ctx.cl_prefill(prompt, tap_hidden=True)
    got = ctx.cl_read_hidden_ring()[0].double().cuda()
    ctx.close()
    x = W["embed"][torch.as_tensor(np.asarray(prompt), device="cuda", dtype=torch.long)].double()
    xn = x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * W["norm2"][0].double()
    up = torch.nn.functional.silu(xn @ W["wg"][0].double().T) * (xn @ W["wu"][0].double().T)
    ffn = up @ W["wd"][0].double().T
    err = got - (x + ffn)
    half = 2.0 ** (-11 if wd == "fp16" else -8)
    assert (err.abs() - half * (x + ffn).abs()).max() <= 1e-4 * ffn.abs().max()
    bias = float((err * ffn).sum() / (ffn * ffn).sum())
    assert abs(bias) <= (5e-6 if wd == "fp16" else 8e-6), bias
