"""Windows at and beyond the sequence (Fig. 2b): a window of nL positions or more, up to the
largest int, hides no key, so a LOCAL call gives the bits of the CROSS call, in both
directions, for full and final-stream queries and for decoding, at every head dim; one
position less hides exactly one pair, which is compared with the oracle."""
import pytest
import torch

import guards
import oracle
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import AttnShape, CROSS, LOCAL

from parity import assert_fwd_close, assert_grads_close, check_status, gpu_fwd_bwd

pytestmark = pytest.mark.gpu

INT_MAX = 2**31 - 1


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _final(q, k, v, do, mode, window):
    qd, kd, vd, dod = q.cuda(), k.cuda(), v.cuda(), do.cuda()
    B, L, Hq, Dh = q.shape
    n, Hkv = k.shape[1] // L, k.shape[2]
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    o, lse = guards.like(qd), guards.empty((B, Hq, L), torch.float32)
    binding.sfa_fwd_final(qd, kd, vd, o, lse, mode, window=window, dev_status=st)
    dq, dk, dv = guards.like(qd), guards.like(kd), guards.like(vd)
    ws = guards.empty((binding.sfa_bwd_final_workspace_bytes(B, L, n, Hq, Hkv, Dh, mode),), torch.uint8)
    binding.sfa_bwd_final(qd, kd, vd, o, lse, dod, dq, dk, dv, mode, ws, window=window, dev_status=st)
    check_status(st)
    return [x.cpu() for x in (o, lse, dq, dk, dv)]


@pytest.mark.parametrize("Dh", [64, 128, 256])
@pytest.mark.parametrize("Hq,Hkv,L,n", [(4, 2, 300, 2), (6, 1, 129, 1), (3, 3, 70, 4)])
def test_window_without_effect(Hq, Hkv, L, n, Dh):
    s = AttnShape(1, L, n, Hq, Hkv, Dh)
    q, k, v, do = inputs.attn_inputs(s, seed=L + Dh)
    full = gpu_fwd_bwd(q, k, v, do, n, CROSS)
    fin = [x[:, n - 1::n].contiguous() for x in (q, do)]
    last = _final(fin[0], k, v, fin[1], CROSS, 0)
    for window in (n * L, n * L + 1, INT_MAX - 300, INT_MAX):
        for a, b in zip(gpu_fwd_bwd(q, k, v, do, n, LOCAL, window=window), full):
            assert torch.equal(a, b), window
        for a, b in zip(_final(fin[0], k, v, fin[1], LOCAL, window), last):
            assert torch.equal(a, b), window
    o, lse, dq, dk, dv = gpu_fwd_bwd(q, k, v, do, n, LOCAL, window=n * L - 1)
    assert_fwd_close(o, lse, *oracle.sfa_fwd(q, k, v, n, LOCAL, None, n * L - 1))
    assert_grads_close([(m, a, r) for m, a, r in zip(("dq", "dk", "dv"), (dq, dk, dv),
                                                     oracle.sfa_bwd(q, k, v, do, n, LOCAL, None, n * L - 1))])


@pytest.mark.parametrize("Dh", [64, 128, 256])
def test_decode_window_without_effect(Dh):
    B, Lcap, n, Hq, Hkv = 2, 90, 3, 4, 2
    q = inputs.normal_bf16((B, n, Hq, Dh), 1).cuda()
    kc = inputs.normal_bf16((B, Lcap * n, Hkv, Dh), 2).cuda()
    vc = inputs.normal_bf16((B, Lcap * n, Hkv, Dh), 3).cuda()
    lens = torch.tensor([90, 41], dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")

    def run(mode, window):
        o = guards.like(q)
        ws = guards.empty((binding.sfa_decode_workspace_bytes(B, Lcap, n, Hq, Hkv, Dh, mode, window),), torch.uint8)
        binding.sfa_decode(q, kc, vc, lens, o, n, mode, ws, window=window, dev_status=st)
        check_status(st)
        return o.clone()

    ref = run(CROSS, 0)
    for window in (n * Lcap, INT_MAX):
        assert torch.equal(run(LOCAL, window), ref), window
