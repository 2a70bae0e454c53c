"""Allocation-free scoring on the tensor cores where its rows do not fit the scratch for their parts at once, and at the lines between
its kernels (run on a B200)."""
import math

import numpy as np
import pytest
import torch

import paper_2604_14612_b200 as cl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,V,d", [(700, 3001, 8192), (513, 1000, 5120), (257, 500, 8192), (130, 449, 72), (12, 200, 4096), (11, 200, 4096),
                                   (5, 32000, 768), (4, 32000, 768), (7, 12288, 1024), (1500, 65, 776)])
def test_calls_in_several_launches(R, V, d):
    """Against fp64.  Activations enter with 26 bits, sums are fp32 with their remainders carried: the largest errors of the kernels' own
    tests are 3e-7 of a confidence's or probability's 2-norm (bound: three times that); heads are chosen so that these are not small against 1."""
    g = torch.Generator(device="cuda").manual_seed(R + V)
    head = (torch.randn((V, d), generator=g, device="cuda") * (1.28 / d ** 0.5)).bfloat16()
    gain = 1.0 + 0.1 * torch.randn((d,), generator=g, device="cuda")
    tok = torch.randint(0, V, (R,), generator=g, device="cuda")
    hidden = (head[tok].float() * (d ** 0.5 / 1.28) * min(0.9, 8.0 / (1.28 * d ** 0.5)) + torch.randn((R, d), generator=g, device="cuda")).bfloat16()
    got = cl.cl_layer_confidences_static(head, gain, hidden[None].contiguous(), rms_eps=1e-5)
    h = hidden.double()
    lg = (h * torch.rsqrt((h * h).mean(-1, keepdim=True) + 1e-5) * gain.double()) @ head.double().T
    lp = torch.log_softmax(lg, -1)
    conf, pmax = 1 + (lp.exp() * lp).sum(-1) / math.log(V), lp.max(-1).values.exp()
    for k, want in (("conf", conf), ("p_max", pmax)):
        w = want.cpu().numpy()
        assert np.linalg.norm(got[k].ravel() - w) <= 1e-6 * np.linalg.norm(w), k
    top = torch.topk(lg, 2, -1)
    clear = (top.values[:, 0] - top.values[:, 1] > 1e-4).cpu().numpy()
    assert (got["argmax"].ravel() == top.indices[:, 0].cpu().numpy())[clear].all()
