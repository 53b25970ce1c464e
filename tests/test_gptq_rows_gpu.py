"""GPU: the row-owner GPTQ encoder at the edges of its tiles, bit-exact with
the oracle on sampled rows (every row's codes depend on that row and the
factor alone).

Every rows-per-block count (8, 16, 28, 32) with a ragged last group, groups in
several waves, every block size (64, 128, 256), column counts that end in each of the
update's segments (512 columns, then 128 or a part), one and more parts of the
sample pairs and of the scan, zero rows (no quotient by the reciprocal) and a factor with
diagonal entries outside the reciprocal's range."""
from fractions import Fraction

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("n,k,b,osr", [(13, 1280, 128, 2), (1003, 768, 128, Fraction(3, 2)), (2403, 256, 128, 2),
                                       (4190, 384, 128, Fraction(5, 2)), (4301, 256, 128, 3), (9801, 256, 64, 2),
                                       (21, 704, 64, 3), (9, 128, 128, 2), (5, 64, 64, Fraction(3, 2)),
                                       (2450, 512, 256, 2), (4309, 768, 256, 3), (11, 512, 256, Fraction(9, 8)),
                                       (6, 192, 64, 7)])
def test_gptq_rows_bit_exact(sdq, q, n, k, b, osr):
    import torch
    assert torch.cuda.is_available()
    rng = np.random.default_rng(n + k + b)
    d = sdq.LayerDesc(n, k, b, Fraction(osr), q)
    signs = np.where(rng.random(b) < 0.5, -1, 1).astype(np.int8)
    plan = sdq.Plan(d, signs)
    w = (rng.standard_normal((n, k)) * 0.02).astype(np.float32)
    w[n // 2] = 0.0
    u = np.triu(rng.standard_normal((k, k)) * 0.1 / np.sqrt(k), 1)
    diag = rng.random(k) + 0.5
    diag[3], diag[k // 2] = 2.0 ** 40, 2.0 ** -35
    u += np.diag(diag)
    u = u.astype(np.float32)
    u[np.tril_indices(k, -1)] = np.nan          # only the upper triangle is used
    codes, alpha = plan.encode_gptq(torch.from_numpy(w).cuda(), torch.from_numpy(u).cuda())
    rows = np.unique(np.concatenate([[0, n - 1, n // 2], rng.integers(0, n, 9)]))
    uo = np.triu(u)
    oc, oa = O.encode_gptq(w[rows], uo, b, d.n_b, q, O.ALPHA_MAXABS, signs)
    assert np.array_equal(alpha.cpu().numpy()[rows], oa)
    got = codes.cpu().numpy().view(np.uint32).reshape(n, -1)[rows]
    assert np.array_equal(got, O.pack_plain(oc, q))
