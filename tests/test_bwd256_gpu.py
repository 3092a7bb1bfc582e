"""The head-dim-256 backward's own branches (derivative of Eq. 4 / Fig. 2, Sec. 3.1):
pairs of 128-row tiles at their edges, query-tile pairs of two heads (even groups) and of
one head (odd groups), head chunks, and the phase-by-phase entry points."""
import math

import pytest
import torch

import guards
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import AttnShape, CROSS, LOCAL, WITHIN

from parity import assert_grads_close, check_status, gpu_fwd, gpu_fwd_bwd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _documented_gradient(q, k, v, o, lse, do, s, mode, window):
    """sfa_bwd's formula in 64 bits for the o and lse it is given: P = exp(scale q k^T - lse),
    dS = P (dO v^T - rowsum(dO o)).  (With two rows the bf16 rounding of o alone moves dq by
    1.1e-2 of its norm against the gradient of the unrounded forward.)"""
    G, N, scale = s.Hq // s.Hkv, s.nL, 1 / math.sqrt(s.Dh)
    Q, O, D = (x.double().permute(0, 2, 1, 3) for x in (q, o, do))
    K, V = (x.double().permute(0, 2, 1, 3).repeat_interleave(G, 1) for x in (k, v))
    p = torch.arange(N)
    vis = p[None, :] <= p[:, None]
    if mode == WITHIN:
        vis &= p[None, :] % s.n == p[:, None] % s.n
    if mode == LOCAL:
        vis &= p[None, :] > p[:, None] - window
    P = torch.exp(scale * Q @ K.transpose(2, 3) - lse.double()[..., None]) * vis
    dS = P * (D @ V.transpose(2, 3) - (D * O).sum(-1, keepdim=True))
    fold = lambda x: x.unflatten(1, (s.Hkv, G)).sum(2).permute(0, 2, 1, 3)  # noqa: E731
    return ((scale * dS @ K).permute(0, 2, 1, 3), fold(scale * dS.transpose(2, 3) @ Q), fold(P.transpose(2, 3) @ D))


# rows of one problem: two rows, both sides of a 128-row tile and of a 256-row pair, a
# second pair of one row; groups of 1, 2 and 3 heads
@pytest.mark.parametrize("rows", [2, 127, 129, 255, 256, 257])
@pytest.mark.parametrize("Hq,Hkv", [(2, 2), (2, 1), (3, 1)])
def test_pair_edges(rows, Hq, Hkv):
    for s, mode, window in ((AttnShape(1, rows, 1, Hq, Hkv, 256), CROSS, 0), (AttnShape(1, rows, 2, Hq, Hkv, 256), WITHIN, 0),
                            (AttnShape(1, rows, 1, Hq, Hkv, 256), LOCAL, 130)):
        q, k, v, do = inputs.attn_inputs(s, seed=rows + 7 * Hq)
        got = gpu_fwd_bwd(q, k, v, do, s.n, mode, 0.0, window)
        ref = _documented_gradient(q, k, v, got[0], got[1], do, s, mode, window)
        assert_grads_close(list(zip(("dq", "dk", "dv"), got[2:], ref)))


@pytest.mark.parametrize("shape,mode", [((1, 200, 2, 4, 2, 256), WITHIN), ((1, 150, 2, 12, 1, 256), CROSS)])
def test_phases_match_whole_call(shape, mode):
    # prep, main and finalize one by one (fp32 dQ through the workspace) against sfa_bwd
    # (dQ as bf16 straight from the main pass): the same fp32 sums, scaled and rounded once,
    # so dQ is the same bits; dK and dV may be summed over another number of head chunks,
    # in fp32: one bf16 rounding apart at most, 2^-8 relative plus the 2^-9 of each side's
    # own fp32 order on cancelling sums, well inside 1e-2 of the norm
    s = AttnShape(*shape)
    q, k, v, do = inputs.attn_inputs(s, seed=17)
    qd, kd, vd, o, lse = gpu_fwd(q, k, v, s.n, mode)
    dod = do.cuda()
    ws = guards.empty((binding.sfa_bwd_workspace_bytes(s.B, s.L, s.n, s.Hq, s.Hkv, s.Dh, mode),), torch.uint8)
    outs = []
    for phased in (False, True):
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        dq, dk, dv = guards.like(qd), guards.like(kd), guards.like(vd)
        if phased:
            binding.sfa_bwd_prep(o, dod, lse, s.n, mode, ws, s.Hkv)
            binding.sfa_bwd_main(qd, kd, vd, dod, dk, dv, s.n, mode, ws, dev_status=st)
            binding.sfa_bwd_finalize(dq, s.n, mode, ws, s.Hkv)
        else:
            binding.sfa_bwd(qd, kd, vd, o, lse, dod, dq, dk, dv, s.n, mode, ws, dev_status=st)
        check_status(st)
        outs.append((dq.cpu(), dk.cpu(), dv.cpu()))
    assert torch.equal(outs[0][0].view(torch.int16), outs[1][0].view(torch.int16))
    assert_grads_close(list(zip(("dk", "dv"), outs[1][1:], outs[0][1:])))
