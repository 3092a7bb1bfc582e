"""dQ written into the buffer of an input of the same call (dout's or q's): the main pass
streams q and dout to other work items until its end, so dQ takes the way through the
workspace there.  Same bits as with a buffer of its own (the same fp32 sums, rounded once); dK
and dV may be summed over another number of head chunks in fp32 and agree to a bf16 rounding,
well inside 1e-2 of the norm.  More work items than SMs, so that some start after others end."""
import pytest
import torch

import guards
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import CROSS, LOCAL, WITHIN

from parity import assert_grads_close, check_status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("final", [False, True])
@pytest.mark.parametrize("Hq,Hkv,Dh,mode,window", [(8, 2, 64, WITHIN, 0), (8, 8, 128, CROSS, 0), (8, 2, 128, LOCAL, 200),
                                                   (6, 2, 256, WITHIN, 0), (4, 4, 256, CROSS, 0)])
def test_dq_in_an_input(Hq, Hkv, Dh, mode, window, final):
    B, L, n = 2, 700, 3
    q = inputs.normal_bf16((B, L if final else n * L, Hq, Dh), Dh).cuda()
    do = inputs.normal_bf16(tuple(q.shape), Dh + 3).cuda()
    k = inputs.normal_bf16((B, n * L, Hkv, Dh), Dh + 1).cuda()
    v = inputs.normal_bf16((B, n * L, Hkv, Dh), Dh + 2).cuda()
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    o, lse = guards.like(q), guards.empty((B, Hq, q.shape[1]), torch.float32)
    if final:
        binding.sfa_fwd_final(q, k, v, o, lse, mode, window=window, dev_status=st)
        ws = binding.sfa_bwd_final_workspace_bytes(B, L, n, Hq, Hkv, Dh, mode)
    else:
        binding.sfa_fwd(q, k, v, o, lse, n, mode, window=window, dev_status=st)
        ws = binding.sfa_bwd_workspace_bytes(B, L, n, Hq, Hkv, Dh, mode)
    ws = guards.empty((ws,), torch.uint8, 255)

    def grads(where):
        qb, dob = q.clone(), do.clone()
        dq = {"own": guards.like(q), "dout": dob, "q": qb}[where]
        dk, dv = guards.like(k), guards.like(v)
        if final:
            binding.sfa_bwd_final(qb, k, v, o, lse, dob, dq, dk, dv, mode, ws, window=window, dev_status=st)
        else:
            binding.sfa_bwd(qb, k, v, o, lse, dob, dq, dk, dv, n, mode, ws, window=window, dev_status=st)
        check_status(st)
        return dq, dk, dv

    ref = grads("own")
    for where in ("dout", "q"):
        got = grads(where)
        assert torch.equal(got[0], ref[0]), where
        assert_grads_close([(m, a.cpu(), b.cpu()) for m, a, b in zip(("dk", "dv"), got[1:], ref[1:])])
