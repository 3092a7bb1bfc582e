"""The backward phase by phase: sfa_bwd_main adds its dQ into the workspace's fp32 accumulator,
which sfa_bwd_prep (or sfa_bwd_clear) zeroes.  One main pass gives sfa_bwd's bits; a second
one without a clear exactly twice the sum, so exactly twice dQ (a power of two, in fp32 and
in bf16); a new prep starts over, over whatever the workspace held."""
import pytest
import torch

import guards
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import AttnShape, CROSS, LOCAL, WITHIN, WITHIN_NAIVE

from parity import check_status, gpu_fwd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("shape,mode,window", [((1, 70, 2, 4, 4, 64), WITHIN, 0), ((2, 150, 1, 6, 2, 64), LOCAL, 40),
                                               ((1, 200, 2, 4, 2, 128), CROSS, 0), ((1, 90, 3, 8, 1, 128), WITHIN_NAIVE, 0),
                                               ((1, 130, 2, 4, 2, 256), WITHIN, 0), ((2, 65, 2, 3, 1, 256), LOCAL, 70)])
def test_main_adds_to_the_accumulator(shape, mode, window):
    s = AttnShape(*shape)
    q, k, v, do = inputs.attn_inputs(s, seed=s.L + s.Dh)
    qd, kd, vd, o, lse = gpu_fwd(q, k, v, s.n, mode, window=window)
    dod = do.cuda()
    dims = (s.B, s.L, s.n, s.Hq, s.Hkv, s.Dh, mode)
    ws = guards.empty((binding.sfa_bwd_workspace_bytes(*dims),), torch.uint8, 255)  # NaN bytes
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    dk, dv = guards.like(kd), guards.like(vd)

    def main_and_dq():
        binding.sfa_bwd_main(qd, kd, vd, dod, dk, dv, s.n, mode, ws, window=window, dev_status=st)
        dq = guards.like(qd)
        binding.sfa_bwd_finalize(dq, s.n, mode, ws, s.Hkv)
        check_status(st)
        return dq

    ref = guards.like(qd)
    ws1 = guards.like(ws)
    binding.sfa_bwd(qd, kd, vd, o, lse, dod, ref, guards.like(kd), guards.like(vd), s.n, mode, ws1, window=window, dev_status=st)
    binding.sfa_bwd_prep(o, dod, lse, s.n, mode, ws, s.Hkv)
    assert torch.equal(main_and_dq(), ref)
    dk1, dv1 = dk.clone(), dv.clone()
    assert torch.equal(main_and_dq(), 2 * ref)
    assert torch.equal(dk, dk1) and torch.equal(dv, dv1)  # overwritten
    binding.sfa_bwd_clear(*dims, ws)
    assert torch.equal(main_and_dq(), ref)
    binding.sfa_bwd_prep(o, dod, lse, s.n, mode, ws, s.Hkv)
    assert torch.equal(main_and_dq(), ref)
