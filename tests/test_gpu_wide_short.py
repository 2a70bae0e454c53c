"""The wide prompt pass of short prompts, and its norm kernel with one, two and four chunks of a row per thread (run on a B200)."""
import dataclasses

import numpy as np
import pytest

import paper_2604_14612_b200 as cl
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,n,wd", [(4160, 65, 150, "bf16"), (4096, 32, 147, "bf16"), (4096, 32, 200, "fp16"), (5120, 40, 160, "bf16"),
                                          (8256, 129, 40, "bf16"), (8256, 129, 160, "fp16"),
                                          (768, 12, 17, "bf16"), (768, 12, 18, "fp16"), (768, 12, 31, "bf16"), (768, 12, 33, "bf16")])
def test_rows_a_thread_and_short_prompts(monkeypatch, d, heads, n, wd):
    """Against the 8-row passes.  Widths over 8192 read part of a row twice.  Both sides keep 16 mantissa bits of the activations and
    round taps to the storage type: taps agree to one bf16 ulp at the top of their range.  Logits (2-norm): a cache entry that one
    side rounds the other way differs by up to 2^-7 of itself; operands off by 2^-17, sums by several of those, do that to one entry
    in 2^6 at most (half a step is 2^-9): sqrt(2^-6) * 2^-7 = 1e-3."""
    sh = dataclasses.replace(synth.WORKLOADS["C2"].shape, n_layers=1, max_seq=n + 16, weight_dtype=wd, vocab=2000, d_model=d, n_heads=heads,
                             n_kv_heads=0, d_ffn=512)
    W = synth.make_weights(sh, 31, device="cuda")
    prompt = synth.make_prompt(31, n, sh.vocab)
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
    assert np.abs(out[0][1]).max() > 0
    assert np.abs(out[0][1] - out[1][1]).max() <= 2 ** -7 * max(1.0, float(np.abs(out[0][1]).max()))
    assert np.linalg.norm(out[0][2] - out[1][2]) <= 1e-3 * np.linalg.norm(out[0][2])
