"""GPU: the code-domain prefill contraction over its tile and split edges.

Batches around the 16-row steps of the batch tile, the 128-row limit of two
thread blocks per SM and the 256-row limit of a tile; k chunks of unequal and
odd stage counts (split over a cluster's thread blocks), K shorter than the
largest split; ragged rows.  Every element within the bf16 bound of its
arithmetic (tests/errbound.py), and the same bits on every call (the cluster
adds its partial sums in a fixed order)."""
from fractions import Fraction

import numpy as np
import pytest

import errbound as EB
import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("m", [65, 112, 113, 128, 129, 255, 257, 400])
@pytest.mark.parametrize("n,k,b,osr", [(130, 128, 128, 1), (7, 1408, 128, Fraction(5, 2)), (513, 1152, 128, 3)])
def test_prefill_split_matches_oracle(sdq, torch_cuda, q, m, n, k, b, osr):
    torch = torch_cuda
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
    assert sdq.sdq_forward_route(plan.handle, m) == 2
    ws = plan.alloc_workspace(m)
    ws.fill_(0xFF)
    y = plan.forward(tiled, al, x, ws=ws)
    y2 = torch.full_like(y, float("nan"))
    sdq.sdq_prep_activations(plan.handle, x, m, ws)
    sdq.sdq_contract(plan.handle, tiled, al, m, y2, ws)
    assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
    assert torch.equal(y, y2)
    xf = W.bf16_to_float(bits)
    yr = O.forward_code_domain(xf, codes, alpha, b, d.n_b, signs)
    EB.check(y.cpu().numpy(), yr, EB.forward_bound(xf, codes, alpha, b, d.n_b, signs), f"M={m} n={n} k={k}")
