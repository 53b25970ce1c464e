"""GPU: the tensor-core prefill prepare kernel over its rule, through the
forward's outputs (each element within the bf16 bound of the route): every
block size it takes (64 .. 512) and the ones it leaves (32, 1024), n_b from
64 to 1536 (one column part and several, the K padding of an odd number of
64-code chunks), few row tiles (64 columns per thread block) and many."""
from fractions import Fraction

import numpy as np
import pytest

import errbound as EB
import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("n,k,b,osr,m", [(40, 192, 64, 1, 65), (130, 960, 64, 3, 700), (20, 8192, 64, 2, 300),
                                         (70, 256, 256, Fraction(3, 2), 77), (33, 2560, 256, Fraction(5, 2), 530),
                                         (50, 512, 512, 3, 100), (17, 2048, 512, 2, 640), (24, 8192, 128, 2, 767),
                                         (24, 640, 128, Fraction(5, 2), 129), (30, 256, 32, 2, 66),
                                         (30, 1024, 1024, 2, 66)])
def test_prefill_prepare_block_sizes(sdq, q, n, k, b, osr, m):
    import torch
    assert torch.cuda.is_available()
    d = sdq.LayerDesc(n, k, b, Fraction(osr), q, 1, 0)
    rng = np.random.default_rng(n + k + m)
    signs = np.where(rng.random(b) < 0.5, -1, 1).astype(np.int8)
    plan = sdq.Plan(d, signs)
    codes = W.random_codes(n, plan.k_eff, q, n + m)
    tiled = plan.pack(torch.from_numpy(O.pack_plain(codes, q).ravel().view(np.int32)).cuda())
    alpha = (rng.random(n) * 0.05 + 0.01).astype(np.float32)
    bits = W.float_to_bf16(rng.standard_normal((m, k)).astype(np.float32))
    x = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    ws = plan.alloc_workspace(m)
    ws.fill_(0xFF)
    y = plan.forward(tiled, torch.from_numpy(alpha).cuda(), x, ws=ws)
    assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
    xf = W.bf16_to_float(bits)
    yr = O.forward_code_domain(xf, codes, alpha, b, d.n_b, signs)
    EB.check(y.cpu().numpy(), yr, EB.forward_bound(xf, codes, alpha, b, d.n_b, signs), f"M={m} B={b}")
