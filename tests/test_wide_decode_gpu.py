"""GPU: decode batches on both sides of the line where they move to the
prefill contraction (M = 24, 40 or 56 by the layer's size), and layers that
stay below it for a rule's sake (blocks of 32, n_b not a multiple of 64): forward, prepare +
contract (the same bits, on a workspace of exactly the bytes asked for, filled
with NaN patterns), the fp32 x_tilde that sdq_read_prep returns, and y +=."""
from fractions import Fraction

import numpy as np
import pytest

import errbound as EB
import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("m", [23, 24, 33, 64])
@pytest.mark.parametrize("n,k,b,osr", [(130, 1152, 128, 3), (1000, 960, 64, 2), (70, 512, 512, 2), (129, 640, 128, Fraction(5, 2)),
                                       (90, 512, 32, 3), (77, 640, 64, Fraction(9, 4))])
def test_wide_decode(sdq, q, m, n, k, b, osr):
    import torch
    assert torch.cuda.is_available()
    d = sdq.LayerDesc(n, k, b, Fraction(osr), q, 1, 0)
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
    ws.fill_(0xFF)
    y = plan.forward(tiled, al, x, ws=ws)
    assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
    ws.fill_(0xFF)
    y2 = torch.full_like(y, float("nan"))
    sdq.sdq_prep_activations(plan.handle, x, m, ws)
    sdq.sdq_contract(plan.handle, tiled, al, m, y2, ws)
    xf = W.bf16_to_float(bits)
    xt = torch.empty((m, plan.k_eff), dtype=torch.float32, device="cuda")
    sdq.sdq_read_prep(plan.handle, m, ws, xt)
    want = O.prep_activations(xf, b, d.n_b, signs)
    assert np.abs(xt.cpu().numpy() - want).max() < 2e-5 * np.abs(want).max()
    sdq.sdq_contract_add(plan.handle, tiled, al, m, y2, ws)
    assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
    yr = O.forward_code_domain(xf, codes, alpha, b, d.n_b, signs)
    bound = EB.forward_bound(xf, codes, alpha, b, d.n_b, signs, T=3)
    EB.check(y.cpu().numpy(), yr, bound, "forward")
    assert np.abs(y2.cpu().numpy() - 2 * y.cpu().numpy()).max() <= 2e-5 * np.abs(yr).max()


@pytest.mark.parametrize("m", [1, 5, 40, 64])
def test_read_prep_after_forward(sdq, m):
    import torch
    n, k, b = 256, 896, 128
    plan = sdq.Plan(sdq.LayerDesc(n, k, b, Fraction(5, 2), O.TERNARY, 1, 0))
    bits = W.float_to_bf16(np.random.default_rng(m).standard_normal((m, k)).astype(np.float32))
    x = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    ws = plan.alloc_workspace(m)
    ws.fill_(0xFF)
    plan.forward(plan.alloc_tiled().zero_(), torch.ones(n, device="cuda"), x, ws=ws)
    xt = torch.empty((m, plan.k_eff), dtype=torch.float32, device="cuda")
    sdq.sdq_read_prep(plan.handle, m, ws, xt)
    want = O.prep_activations(W.bf16_to_float(bits), b, b * 5 // 2, None)
    assert np.abs(xt.cpu().numpy() - want).max() < 2e-5 * np.abs(want).max()
