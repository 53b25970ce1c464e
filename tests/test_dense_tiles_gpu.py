"""GPU: the dense route's tiles: batches around multiples of its batch tiles
(one and two weight tiles per pair of thread blocks; the last two shapes end
in a wave of single tiles on devices of 70 to 76 such pairs), rows
that end inside a tile (the rebuilt weights' stores are clipped there) and
every number of 64-code chunks per block (one and two epilogue buffers), each
element within the bound of the rebuilt weights' bf16 rounding."""
from fractions import Fraction

import numpy as np
import pytest

import errbound as EB
import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("n,k,osr,m", [(1, 128, 2, 768), (130, 256, Fraction(3, 2), 769), (257, 384, Fraction(5, 2), 1040),
                                       (4200, 128, 3, 800), (5000, 128, 1, 1601), (2600, 256, 2, 2305),
                                       (6529, 128, 2, 1295), (3713, 128, Fraction(3, 2), 2681)])
def test_dense_tiles(sdq, q, n, k, osr, m):
    import torch
    assert torch.cuda.is_available()
    d = sdq.LayerDesc(n, k, 128, Fraction(osr), q, 1, 0)
    rng = np.random.default_rng(n + k + m)
    signs = np.where(rng.random(128) < 0.5, -1, 1).astype(np.int8)
    plan = sdq.Plan(d, signs)
    assert sdq.sdq_forward_route(plan.handle, m) == 3
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
    yr = O.forward_code_domain(xf, codes, alpha, 128, d.n_b, signs)
    EB.check(y.cpu().numpy(), yr, EB.forward_bound(xf, codes, alpha, 128, d.n_b, signs, dense=True), f"M={m} n={n}")
