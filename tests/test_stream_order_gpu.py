"""GPU: a forward's inputs may come from the kernels just before it in the
stream, from this library's own too, which let the kernels behind them start
early: its scales, codes and activations are read after those have written
them.

A long contraction of few thread blocks (the chip has room for the next call
beside it) writes y; the next call, with nothing between them, takes that y
as its scales or as the bits of its codes, and gives what it gives once the
stream has been waited for."""
from fractions import Fraction

import pytest

pytestmark = pytest.mark.gpu

M0, N0, K0 = 65, 128, 1 << 16      # the writer: 8 thread blocks
B = 128


def _codes(torch, plan, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = torch.randint(-2 ** 31, 2 ** 31, (plan.alloc_tiled().numel(),), generator=g, device="cuda", dtype=torch.int32)
    return s & 0x55555555          # 0 and +1


@pytest.mark.parametrize("m", [1, 4, 16, 30])
@pytest.mark.parametrize("call", ["forward", "contract", "contract_add"])
@pytest.mark.parametrize("what", ["alpha", "codes"])
@pytest.mark.parametrize("n,k", [(128, 512), (256, 2048)])
def test_inputs_from_the_kernel_before(sdq, m, call, what, n, k):
    import torch
    assert torch.cuda.is_available()
    g = torch.Generator(device="cuda").manual_seed(n + m)
    first = sdq.Plan(sdq.LayerDesc(N0, K0, B, Fraction(2), 2))
    plan = sdq.Plan(sdq.LayerDesc(n, k, B, Fraction(2), 2))
    t0, a0 = _codes(torch, first, 1), torch.full((N0,), 0.01, device="cuda")
    x0 = torch.randn((M0, K0), generator=g, device="cuda").to(torch.bfloat16)
    ws0, ws = first.alloc_workspace(M0), plan.alloc_workspace(m)
    need = n if what == "alpha" else plan.alloc_tiled().numel()
    y0 = torch.full((max(need, M0 * N0),), 0.5, device="cuda")
    tiled = _codes(torch, plan, 2)
    alpha = torch.rand(n, generator=g, device="cuda") + 0.5
    x = torch.randn((m, k), generator=g, device="cuda").to(torch.bfloat16)

    def second(y):
        al = y0[:n] if what == "alpha" else alpha
        co = y0.view(torch.int32)[:need] if what == "codes" else tiled
        if call == "forward":
            sdq.sdq_linear_forward(plan.handle, co, al, x, m, y, ws)
        else:
            sdq.sdq_prep_activations(plan.handle, x, m, ws)
            getattr(sdq, "sdq_" + call)(plan.handle, co, al, m, y, ws)

    want, y = torch.zeros((m, n), device="cuda"), torch.empty((m, n), device="cuda")
    sdq.sdq_linear_forward(first.handle, t0, a0, x0, M0, y0, ws0)
    torch.cuda.synchronize()
    second(want)
    torch.cuda.synchronize()
    assert torch.isfinite(want).all() and want.abs().max() > 0
    for i in range(4):
        y0[:M0 * N0].fill_(0.25)
        y.zero_()
        torch.cuda.synchronize()
        sdq.sdq_linear_forward(first.handle, t0, a0, x0, M0, y0, ws0)
        second(y)
        torch.cuda.synchronize()
        # (forward, contract_add: split-K sums in an order that is not fixed)
        assert (y - want).abs().max() <= 2e-6 * want.abs().max(), i
