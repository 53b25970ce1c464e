"""GPU: decode batches on both sides of the line where they move to the
prefill contraction (M = 24 up to 40 million codes, 40 up to 200 million, 56
above), and layers that stay below it for a rule's sake (blocks of 32, n_b not
a multiple of 64): forward, prepare + contract (the same bits every time, and
those of forward on the prefill contraction, on a workspace of exactly the
bytes asked for, filled with NaN patterns), the fp32 x_tilde that
sdq_read_prep returns, and y +=."""
from fractions import Fraction

import numpy as np
import pytest

import errbound as EB
import oracle as O
from paper_2510_03275_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _wide(d, m, k_eff):
    """Whether the layer's batch m contracts with the prefill kernel."""
    codes = d.n_out * k_eff
    line = 24 if codes <= 40_000_000 else 40 if codes <= 200_000_000 else 56
    return 64 <= d.block <= 512 and d.n_b % 64 == 0 and m >= line


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
    for i in range(3):
        ws.fill_(0xFF)
        y2 = torch.full_like(y, float("nan"))
        sdq.sdq_prep_activations(plan.handle, x, m, ws)
        sdq.sdq_contract(plan.handle, tiled, al, m, y2, ws)
        assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
        if i == 0:
            y1 = y2
        assert torch.equal(y1, y2)
    wide = _wide(d, m, plan.k_eff)
    if wide:
        assert torch.equal(y, y2)
    xf = W.bf16_to_float(bits)
    xt = torch.empty((m, plan.k_eff), dtype=torch.float32, device="cuda")
    sdq.sdq_read_prep(plan.handle, m, ws, xt)
    want = O.prep_activations(xf, b, d.n_b, signs)
    assert np.abs(xt.cpu().numpy() - want).max() < 2e-5 * np.abs(want).max()
    yr = O.forward_code_domain(xf, codes, alpha, b, d.n_b, signs)
    bound = EB.forward_bound(xf, codes, alpha, b, d.n_b, signs, T=None if wide else 3)
    EB.check(y.cpu().numpy(), yr, bound, "forward")
    EB.check(y1.cpu().numpy(), yr, bound, "contract")
    y2 = y1.clone()
    sdq.sdq_contract_add(plan.handle, tiled, al, m, y2, ws)
    assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
    assert np.abs(y2.cpu().numpy() - 2 * y.cpu().numpy()).max() <= 2e-5 * np.abs(yr).max()


@pytest.mark.parametrize("q", [O.TERNARY, O.BINARY])
@pytest.mark.parametrize("n,k,b,osr,ms", [(2401, 8192, 128, 2, (23, 24)), (5003, 8192, 128, 2, (24, 33, 39, 40)),
                                          (4100, 11008, 64, 3, (39, 40)), (5003, 8192, 512, Fraction(3, 2), (24, 40)),
                                          (14001, 8192, 128, 2, (24, 40, 55, 56)), (17001, 8192, 128, Fraction(3, 2), (55, 56))])
def test_lines_of_larger_layers(sdq, q, n, k, b, osr, ms):
    """Both sides of each line, on layers of the codes it is for (random codes in
    a sample of the rows, zero fields in the others; every output checked)."""
    import torch
    d = sdq.LayerDesc(n, k, b, Fraction(osr), q, 1, 0)
    rng = np.random.default_rng(n + k)
    signs = np.where(rng.random(b) < 0.5, -1, 1).astype(np.int8)
    plan = sdq.Plan(d, signs)
    rows = np.unique(np.concatenate([[0, 127, 128, n - 1], rng.integers(0, n, 20)]))
    codes = W.random_codes(len(rows), plan.k_eff, q, n)
    plain = plan.alloc_plain().zero_()
    plain.view(n, -1)[torch.from_numpy(rows).cuda()] = torch.from_numpy(O.pack_plain(codes, q).view(np.int32)).cuda()
    tiled = plan.pack(plain)
    alpha = (rng.random(n) * 0.05 + 0.01).astype(np.float32)
    al = torch.from_numpy(alpha).cuda()
    rest = np.setdiff1d(np.arange(n), rows)
    for m in ms:
        wide = _wide(d, m, plan.k_eff)
        bits = W.float_to_bf16(rng.standard_normal((m, k)).astype(np.float32))
        x = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
        ws = plan.alloc_workspace(m)
        ws.fill_(0xFF)
        y = plan.forward(tiled, al, x, ws=ws)
        assert sdq.sdq_workspace_status(plan.handle, m, ws) == 0
        ys = []
        for _ in range(2):
            ws.fill_(0xFF)
            ys.append(torch.full_like(y, float("nan")))
            sdq.sdq_prep_activations(plan.handle, x, m, ws)
            sdq.sdq_contract(plan.handle, tiled, al, m, ys[-1], ws)
        assert torch.equal(ys[0], ys[1])
        if wide:
            assert torch.equal(y, ys[0])
        xf = W.bf16_to_float(bits)
        yr = O.forward_code_domain(xf, codes, alpha[rows], b, d.n_b, signs)
        bound = EB.forward_bound(xf, codes, alpha[rows], b, d.n_b, signs, T=None if wide else 3)
        for got, what in ((y, "forward"), (ys[0], "contract")):
            EB.check(got.cpu().numpy()[:, rows], yr, bound, f"{what} M={m}")
        if q == O.TERNARY:
            assert not y.cpu().numpy()[:, rest].any()
        else:        # every code -1: the same sum for every row, up to its scale
            s = y.cpu().numpy()[:, rest] / alpha[rest]
            want = -O.prep_activations(xf, b, d.n_b, signs).sum(axis=1, keepdims=True)
            ones = EB.forward_bound(xf, np.ones((1, plan.k_eff)), np.ones(1), b, d.n_b, signs, T=None if wide else 3)
            assert (np.abs(s - want) <= np.asarray(ones) + 1e-6 * np.abs(s)).all()


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
