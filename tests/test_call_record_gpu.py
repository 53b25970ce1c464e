"""GPU: a timeout of the kernel that prepares a contraction's operand reaches
sdq_workspace_status.  Nothing here times out: what such a kernel leaves in the
workspace's call record (words 2 and 3: the last prepare kernel that gave up and
the last that ran) is written there by the host."""
from fractions import Fraction

import pytest

pytestmark = pytest.mark.gpu

OK, TIMEOUT = 0, -5


def _record(ws, m):
    """The call record: at the start of the workspace of a decode batch that
    contracts with the prefill kernel, in the last 256 bytes of a larger one's."""
    import torch
    return (ws[:32] if m <= 64 else ws[-256:-224]).view(torch.int64)


# prep_tc_kernel (blocks of 128) behind both kinds of workspace, and prep_kernel (blocks of 32), which has no waits
@pytest.mark.parametrize("n,k,b,m", [(256, 512, 128, 30), (256, 512, 128, 100), (256, 512, 32, 100), (256, 512, 128, 800)])
def test_prepare_timeout_is_reported(sdq, n, k, b, m):
    import torch
    assert torch.cuda.is_available()
    plan = sdq.Plan(sdq.LayerDesc(n, k, b, Fraction(2), 2))
    x = torch.randn((m, k), device="cuda").to(torch.bfloat16)
    tiled, alpha = plan.alloc_tiled().zero_(), torch.ones(n, device="cuda")
    y = torch.empty((m, n), device="cuda")
    ws = plan.alloc_workspace(m)
    rec = _record(ws, m)

    def status():
        return sdq.sdq_workspace_status(plan.handle, m, ws)

    def contract():
        sdq.sdq_contract(plan.handle, tiled, alpha, m, y, ws)

    for fill in (0, 0xFF):
        ws.fill_(fill)
        sdq.sdq_prep_activations(plan.handle, x, m, ws)
        contract()
        assert status() == OK
        rec[2] = rec[3].clone()        # the prepare kernel gave up
        contract()
        assert status() == TIMEOUT
        contract()                     # its x_tilde is still what this reads
        assert status() == TIMEOUT
        sdq.sdq_prep_activations(plan.handle, x, m, ws)
        contract()
        assert status() == OK
        rec[2] = rec[3].clone()        # an earlier call's: the forward prepares its own operand
        plan.forward(tiled, alpha, x, ws=ws)
        assert status() == OK
        ran = rec.clone()
        assert int(ran[3]) >> 47 == 1 and int(ran[1]) >> 47 == 1 and int(ran[2]) != int(ran[3])
