"""GPU: layout conversions at the edges of their kernels' tiles, bit-exact
against the oracle: rows around a 128-row tile, group counts around a block's
8 groups (plain <-> tiled), and rows around one and several runs of 32 groups
of 80 codes (plain <-> base-3), with more runs than one step of the persistent
grid (1, 2 and 6 runs a row) in the last cases."""
from fractions import Fraction

import numpy as np
import pytest

import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


def _plain(torch, codes, q):
    return torch.from_numpy(O.pack_plain(codes, q).reshape(-1).view(np.int32)).cuda()


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("n,keff", [(127, 448), (128, 512), (129, 576), (257, 1088), (1, 64)])
def test_pack_unpack_tile_edges(sdq, torch_cuda, q, n, keff):
    torch = torch_cuda
    plan = sdq.Plan(sdq.LayerDesc(n, keff, 64, Fraction(1), q))
    codes = W.random_codes(n, keff, q, n + keff)
    plain = _plain(torch, codes, q)
    tiled = torch.full((sdq.sdq_tiled_bytes(plan.desc) // 4,), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
    sdq.sdq_pack(plan.handle, plain, tiled)
    want = O.pack_tiled(codes, q).reshape(-1)
    assert np.array_equal(tiled.cpu().numpy().view(np.uint32), want)
    back = torch.full_like(plain, -1)
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    sdq.sdq_unpack(plan.handle, tiled, back, bad)
    assert torch.equal(back, plain) and int(bad.item()) == 0


@pytest.mark.parametrize("n,keff", [(3, 2496), (5, 2560), (2, 2624), (9, 5184), (1, 64), (6500, 2624),
                                    (20001, 64), (2001, 12864)])
def test_base3_run_edges(sdq, torch_cuda, n, keff):
    torch = torch_cuda
    plan = sdq.Plan(sdq.LayerDesc(n, keff, 64, Fraction(1), O.TERNARY))
    codes = W.random_codes(n, keff, O.TERNARY, n + keff)
    plain = _plain(torch, codes, O.TERNARY)
    b3 = torch.full((sdq.sdq_base3_bytes(plan.desc),), 0x5A, dtype=torch.uint8, device="cuda")
    sdq.sdq_pack_base3(plan.handle, plain, b3)
    assert np.array_equal(b3.cpu().numpy().reshape(n, -1), O.pack_base3(codes))
    back = torch.full_like(plain, -1)
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    sdq.sdq_unpack_base3(plan.handle, b3, back, bad)
    assert torch.equal(back, plain) and int(bad.item()) == 0
