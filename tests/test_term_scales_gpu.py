"""GPU: the e2m1 terms of activations of every magnitude, those whose terms'
scales reach the smallest power of two among them, from both writers of the
terms (the prepare kernel's image where n_b is a multiple of 64, the
contraction's own writer elsewhere).

Row r's only code is +1 at place r, so y is x_tilde as the terms hold it; it
is compared with the fp32 x_tilde that sdq_read_prep returns.  The last of T
terms is rounded by at most half a unit of its scale 2^(e - 3 (T - 1)): 0.25 x
8^-(T-1) of the group's maximum (of its 128-code block's, at most), or 2^-127
where that scale is the smallest there is, 2^-126."""
from fractions import Fraction

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 8, 20])
@pytest.mark.parametrize("b,osr,k", [(64, 2, 256), (16, Fraction(5, 2), 192)])
@pytest.mark.parametrize("shift", [0, -90, -112, -118, -122, -126, -130, 120])
def test_terms_of_every_magnitude(sdq, m, b, osr, k, shift):
    import torch
    assert torch.cuda.is_available()
    n = int(k * osr)
    plan = sdq.Plan(sdq.LayerDesc(n, k, b, Fraction(osr), O.TERNARY))
    codes = np.eye(n, dtype=np.int8)
    tiled = plan.pack(torch.from_numpy(O.pack_plain(codes, O.TERNARY).ravel().view(np.int32)).cuda())
    scale = -100 if shift > 0 else 60
    alpha = torch.full((n,), 2.0 ** scale, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(m)
    x = torch.randint(-7, 8, (m, k), generator=g, device="cuda").double() * 2.0 ** shift
    x[:, :2 * b] *= 2.0 ** -3                       # (groups of different magnitudes)
    x[:, 3 * b:4 * b] = 0.0
    x = x.to(torch.bfloat16)
    ws = plan.alloc_workspace(m)
    y = torch.empty((m, n), device="cuda")
    sdq.sdq_prep_activations(plan.handle, x, m, ws)
    sdq.sdq_contract(plan.handle, tiled, alpha, m, y, ws)
    xt = torch.empty((m, n), device="cuda")
    sdq.sdq_read_prep(plan.handle, m, ws, xt)
    xt = xt.cpu().numpy().astype(np.float64)
    got = y.cpu().numpy().astype(np.float64) * 2.0 ** -scale
    terms = 6 if m <= 4 else 4 if m <= 16 else 3
    pad = np.zeros((m, -(-n // 128) * 128))
    pad[:, :n] = np.abs(xt)
    top = np.repeat(pad.reshape(m, -1, 128).max(axis=2), 128, axis=1)[:, :n]
    bound = np.maximum(0.25 * 8.0 ** -(terms - 1) * top, 2.0 ** -127) + 2.0 ** -23 * np.abs(xt)
    assert np.isfinite(got).all()
    d = np.abs(got - xt)
    assert (d <= bound).all(), (d / bound).max()
