"""All-layer scoring at the edges of its row blocks, single CTAs and CTA pairs (run on a B200)."""
import numpy as np
import pytest
import torch

import paper_2604_14612_b200 as cl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
def test_scoring_at_block_edges_against_fp64(dtype):
    """One context, row counts on both sides of every block edge (128 rows a CTA, 256 a pair), large before small so that a later
    call uses scratch that an earlier one sized.  Rows are normalised to the storage type (2^-9 / 2^-12 relative an element):
    over 512 elements a logit of spread 2 moves by about 2 * 2^-9 / sqrt(3), 2.3e-3, and the probability and the confidence by at
    most a few times that; the bound is the 1e-2 of the other parity tests."""
    V, d = 5003, 512
    dt = {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator(device="cuda").manual_seed(31)
    head = (torch.randn((V, d), generator=g, device="cuda") * 2 / d ** 0.5).to(dt)
    gain = 1.0 + 0.1 * torch.randn((d,), generator=g, device="cuda")
    ctx = cl.Context(2, d, d // 64, 64, V, 8, dtype)
    ctx.cl_load(dict(lm_head=head, final_norm=gain), head_only=True)
    for R in (2500, 1, 127, 128, 129, 255, 256, 257, 384, 513, 2048):
        hidden = (3 * torch.randn((R, 1, d), generator=g, device="cuda")).to(dt)
        got = ctx.cl_layer_confidences(hidden)
        x = hidden[:, 0].double()
        lg = (x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * gain.double()) @ head.double().T
        lp = torch.log_softmax(lg, -1)
        conf = (1 + (lp.exp() * lp).sum(-1) / np.log(V)).cpu().numpy()
        assert np.abs(got["conf"][:, 0] - conf).max() <= 1e-2, R
        assert np.abs(got["p_max"][:, 0] - lp.max(-1).values.exp().cpu().numpy()).max() <= 1e-2, R
        top = torch.topk(lg, 2).values
        clear = ((top[:, 0] - top[:, 1]) > 5e-2).cpu().numpy()
        assert np.array_equal(got["argmax"][clear, 0], lg.argmax(-1).cpu().numpy()[clear]), R


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
def test_scoring_of_wide_rows_at_block_edges_against_fp64(dtype):
    """Width 4096, where row counts that fill them go to CTA pairs (narrower rows stay with single CTAs): the same bounds, since a
    logit's spread does not depend on the width."""
    V, d = 5003, 4096
    dt = {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator(device="cuda").manual_seed(32)
    head = (torch.randn((V, d), generator=g, device="cuda") * 2 / d ** 0.5).to(dt)
    gain = 1.0 + 0.1 * torch.randn((d,), generator=g, device="cuda")
    ctx = cl.Context(2, d, d // 64, 64, V, 8, dtype)
    ctx.cl_load(dict(lm_head=head, final_norm=gain), head_only=True)
    for R in (2500, 1, 128, 129, 255, 256, 257, 513):
        hidden = (3 * torch.randn((R, 1, d), generator=g, device="cuda")).to(dt)
        got = ctx.cl_layer_confidences(hidden)
        x = hidden[:, 0].double()
        lg = (x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * gain.double()) @ head.double().T
        lp = torch.log_softmax(lg, -1)
        conf = (1 + (lp.exp() * lp).sum(-1) / np.log(V)).cpu().numpy()
        assert np.abs(got["conf"][:, 0] - conf).max() <= 1e-2, R
        assert np.abs(got["p_max"][:, 0] - lp.max(-1).values.exp().cpu().numpy()).max() <= 1e-2, R
        top = torch.topk(lg, 2).values
        clear = ((top[:, 0] - top[:, 1]) > 5e-2).cpu().numpy()
        assert np.array_equal(got["argmax"][clear, 0], lg.argmax(-1).cpu().numpy()[clear]), R
