"""Windowed final-stream problems whose query step (n positions) is wider than the window, so
that some key tiles are seen by no query: between the two query tiles of a forward CTA (odd
head groups: consecutive tiles of one head) and between query tiles of the backward.  Gaps
of none, one and many key tiles, the second query tile full, ragged and of one row, with
the K/V ring passed several times, at every head dim; against the oracle.

Tolerances as for the other final-stream problems: max|dO| <= 2e-2, max|dLSE| <= 1e-3,
gradients rel-L2 <= 1e-2."""
import pytest
import torch

import guards
import oracle
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import LOCAL

from parity import assert_fwd_close, assert_grads_close, check_status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("Dh", [64, 128, 256])
@pytest.mark.parametrize("Hq,Hkv,L,n,window", [
    (1, 1, 300, 128, 1),   # tiles meet without a gap
    (1, 1, 129, 129, 1),   # one tile of gap, the second query tile has one row
    (2, 2, 200, 160, 8),
    (3, 1, 260, 200, 20),  # two CTAs, the second with one query tile of 4 rows
    (1, 1, 256, 256, 128),
    (1, 1, 200, 256, 200),  # a window of more than one tile, no gap
    (2, 1, 200, 256, 1),    # even group: both tiles are the same rows of two heads
])
def test_gap_between_query_tiles(Hq, Hkv, L, n, window, Dh):
    q = inputs.normal_bf16((1, L, Hq, Dh), L + n)
    k = inputs.normal_bf16((1, n * L, Hkv, Dh), L + n + 1)
    v = inputs.normal_bf16((1, n * L, Hkv, Dh), L + n + 2)
    do = inputs.normal_bf16((1, L, Hq, Dh), L + n + 3)
    qd, kd, vd, dod = q.cuda(), k.cuda(), v.cuda(), do.cuda()
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    o, lse = guards.like(qd), guards.empty((1, Hq, L), torch.float32)
    binding.sfa_fwd_final(qd, kd, vd, o, lse, LOCAL, window=window, dev_status=st)
    check_status(st)
    o_ref, lse_ref = oracle.sfa_fwd_final(q, k, v, n, LOCAL, window=window)
    assert_fwd_close(o.cpu(), lse.cpu(), o_ref, lse_ref)

    dq, dk, dv = guards.like(qd), guards.like(kd), guards.like(vd)
    ws = guards.empty((binding.sfa_bwd_final_workspace_bytes(1, L, n, Hq, Hkv, Dh, LOCAL),), torch.uint8)
    binding.sfa_bwd_final(qd, kd, vd, o, lse, dod, dq, dk, dv, LOCAL, ws, window=window, dev_status=st)
    check_status(st)
    dq_ref, dk_ref, dv_ref = oracle.sfa_bwd_final(q, k, v, do, n, LOCAL, window=window)
    if window == 1:  # one visible key: softmax 1, dS = 0, the exact dQ and dK are zero
        assert float(dq.float().abs().max()) <= 1e-5 and float(dk.float().abs().max()) <= 1e-5
        assert_grads_close([("dv", dv.cpu(), dv_ref)])
    else:
        assert_grads_close([(m, a.cpu(), r) for m, a, r in zip(("dq", "dk", "dv"), (dq, dk, dv),
                                                               (dq_ref, dk_ref, dv_ref))])
