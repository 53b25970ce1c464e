"""GPU: the tile encoder at the edges of its rule and its tiles, codes and
alpha bit-exact with the oracle's canonical fp32 encoder.

The tile encoder takes blocks of at least 16 inputs whose codes fill whole
32-bit words, with half its table in shared memory (up to 192 sample pairs) or
read from global memory; the others stay with the row encoder.
Both sides of each line, one computation of the samples for alpha and scan
(the group's blocks fit in one tile) and two (more blocks than virtual rows
in a tile), rows that do not fill the last group, every pair count per lane
(1 .. 6), K_eff that leaves padding words."""
from fractions import Fraction

import numpy as np
import pytest

import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(5, 32, 16, 2), (9, 48, 16, 1), (33, 192, 64, 1), (7, 320, 64, Fraction(3, 2)), (161, 128, 64, 3),
          (3, 8192, 64, 2), (2, 20480, 128, 1), (17, 384, 128, Fraction(3, 2)), (700, 256, 128, 2),
          (1, 18560, 128, 2), (6, 896, 128, Fraction(5, 2)), (5, 640, 128, 3), (4, 256, 128, Fraction(7, 2)),
          (6, 384, 128, Fraction(9, 8)), (3, 512, 256, Fraction(3, 2)), (35, 768, 256, 2), (3, 2048, 256, 3),
          (5, 1024, 512, 2), (20, 1536, 512, Fraction(5, 2)), (2, 512, 512, 3), (3, 1024, 1024, 2), (6, 64, 8, 2),
          (5, 640, 64, 5)]


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("am", [O.ALPHA_MAXABS, O.ALPHA_MEANABS])
@pytest.mark.parametrize("n,k,b,osr", SHAPES)
def test_encode_tile_bit_exact(sdq, q, am, n, k, b, osr):
    import torch
    assert torch.cuda.is_available()
    d = sdq.LayerDesc(n, k, b, Fraction(osr), q, 1, am)
    rng = np.random.default_rng(n + k + b)
    signs = np.where(rng.random(b) < 0.5, -1, 1).astype(np.int8)
    w = (rng.standard_normal((n, k)) * 0.02).astype(np.float32)
    w[0, : b] = 0.0
    plan = sdq.Plan(d, signs)
    codes, alpha = plan.encode(torch.from_numpy(w).cuda())
    oc, oa = O.encode(w, b, d.n_b, q, am, signs)
    assert np.array_equal(alpha.cpu().numpy(), oa)
    got = codes.cpu().numpy().view(np.uint32).reshape(n, -1)
    assert np.array_equal(got, O.pack_plain(oc, q))
