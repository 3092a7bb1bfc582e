"""Programmatic launches of the attention kernels: a chain of dependent calls (each reads what
the one before wrote, or overwrites what it read) enqueued without a host wait gives the bits
of the same chain with a synchronisation after every call, at grids on both sides of one CTA
per SM and of the largest grid that is launched early."""
import pytest
import torch

import guards
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import AttnShape, CROSS

from parity import check_status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _chain(s, q, k, v, do, sync):
    wait = torch.cuda.synchronize if sync else (lambda: None)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    q, k, v, do = (x.clone() for x in (q, k, v, do))
    o, dq, dk, dv = guards.like(q), guards.like(q), guards.like(k), guards.like(v)
    lse = guards.empty((s.B, s.Hq, s.nL), torch.float32)
    ws = guards.empty((binding.sfa_bwd_workspace_bytes(s.B, s.L, s.n, s.Hq, s.Hkv, s.Dh, CROSS),), torch.uint8)
    torch.cuda.synchronize()
    for _ in range(4):  # the gradients are the next layer's operands, the output its gradient
        binding.sfa_fwd(q, k, v, o, lse, s.n, CROSS, dev_status=st)
        wait()
        binding.sfa_bwd(q, k, v, o, lse, do, dq, dk, dv, s.n, CROSS, ws, dev_status=st)
        wait()
        q, dq, k, dk, v, dv, do, o = dq, q, dk, k, dv, v, o, do
    torch.cuda.synchronize()
    check_status(st)
    return [x.view(torch.int16).cpu() for x in (q, k, v, do)] + [lse.view(torch.int32).cpu()]


# forward grids: one CTA per sequence (two at head dim 256, a pair)
@pytest.mark.parametrize("B,Dh", [(1, 64), (152, 64), (153, 128), (304, 128), (1216, 128), (1217, 128),
                                  (1, 256), (76, 256), (77, 256), (608, 256), (609, 256)])
def test_chain_without_host_waits(B, Dh):
    s = AttnShape(B, 24, 1, 2, 1, Dh)
    ins = [x.cuda() for x in inputs.attn_inputs(s, seed=B + Dh)]
    for x, y in zip(_chain(s, *ins, False), _chain(s, *ins, True)):
        assert torch.equal(x, y)
