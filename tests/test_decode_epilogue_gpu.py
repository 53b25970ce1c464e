"""GPU: decode batches at the edges of the one-pipeline epilogue's column
chunks (24 accumulator columns per wait at 3 and 6 terms a row, 32 at 4; the
last chunk whole, ragged, and clamped inside the N columns), of the first
stages' early expansion (fewer stages than expander sets, ragged stages) and of
the streamed B rows, every element within its bound, and the same call on a
workspace of other contents."""
from fractions import Fraction

import numpy as np
import pytest

import errbound as EB
import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("n,k,osr,m", [(130, 256, 2, 3), (130, 256, 2, 4), (257, 768, Fraction(5, 2), 5),
                                       (257, 768, Fraction(5, 2), 8), (768, 768, Fraction(5, 2), 9),
                                       (768, 768, Fraction(5, 2), 16), (768, 384, 2, 17), (300, 1024, 2, 22),
                                       (300, 1024, Fraction(3, 2), 23), (129, 128, 1, 16), (129, 128, 1, 1)])
def test_decode_epilogue_edges(sdq, q, n, k, osr, m):
    import torch
    assert torch.cuda.is_available()
    b = 128
    d = sdq.LayerDesc(n, k, b, Fraction(osr), q)
    rng = np.random.default_rng(n + k + m)
    signs = np.where(rng.random(b) < 0.5, -1, 1).astype(np.int8)
    plan = sdq.Plan(d, signs)
    codes = W.random_codes(n, plan.k_eff, q, n + m)
    tiled = plan.pack(torch.from_numpy(O.pack_plain(codes, q).ravel().view(np.int32)).cuda())
    alpha = (rng.random(n) * 0.05 + 0.01).astype(np.float32)
    al = torch.from_numpy(alpha).cuda()
    bits = W.float_to_bf16(rng.standard_normal((m, k)).astype(np.float32))
    x = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    ws = plan.alloc_workspace(m)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    terms = sdq.sdq_decode_launch_shape(d, m, sms)["T"]
    xf = W.bf16_to_float(bits)
    yr = O.forward_code_domain(xf, codes, alpha, b, d.n_b, signs)
    bound = EB.forward_bound(xf, codes, alpha, b, d.n_b, signs, T=terms)
    for fill in (0xFF, 0x00):
        ws.fill_(fill)
        y = plan.forward(tiled, al, x, ws=ws)
        assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
        EB.check(y.cpu().numpy(), yr, bound, "forward")
    y2 = torch.full_like(y, float("nan"))
    sdq.sdq_prep_activations(plan.handle, x, m, ws)
    sdq.sdq_contract(plan.handle, tiled, al, m, y2, ws)
    EB.check(y2.cpu().numpy(), yr, bound, "contract")
