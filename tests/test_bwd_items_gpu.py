"""The head-dim-64 / 128 backward's work items (derivative of Eq. 4 / Fig. 2, Sec. 3.1): key
and query tiles at their edges, ring laps, head chunks through the space of the fp32 dQ, the
naive intra-stream schedule, and the phase-by-phase entry points."""
import pytest
import torch

import guards
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import AttnShape, CROSS, LOCAL, WITHIN, WITHIN_NAIVE

from parity import assert_grads_close, check_status, gpu_fwd, gpu_fwd_bwd
from test_bwd256_gpu import _documented_gradient

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


# rows of one problem: both sides of a tile, and of a lap of the three- and two-slot rings
# (six and four at head dim 64); one and three heads per K/V head
@pytest.mark.parametrize("rows", [127, 128, 129, 257, 385, 513, 897])
@pytest.mark.parametrize("Hq", [1, 3])
@pytest.mark.parametrize("Dh", [64, 128])
def test_tile_edges(rows, Hq, Dh):
    for s, mode, window in ((AttnShape(1, rows, 1, Hq, 1, Dh), CROSS, 0), (AttnShape(1, rows, 1, Hq, 1, Dh), LOCAL, 130)):
        q, k, v, do = inputs.attn_inputs(s, seed=rows + 7 * Hq)
        got = gpu_fwd_bwd(q, k, v, do, s.n, mode, 0.0, window)
        ref = _documented_gradient(q, k, v, got[0], got[1], do, s, mode, window)
        assert_grads_close(list(zip(("dq", "dk", "dv"), got[2:], ref)))


@pytest.mark.parametrize("shape,mode", [((1, 200, 2, 4, 2, 128), WITHIN), ((1, 150, 2, 12, 1, 64), CROSS),
                                        ((1, 150, 3, 8, 1, 128), WITHIN_NAIVE)])
def test_phases_match_whole_call(shape, mode):
    # prep, main and finalize one by one (fp32 dQ through the workspace) against sfa_bwd (dQ
    # as bf16 straight from the main pass): the same fp32 sums, scaled and rounded once, so
    # dQ is the same bits; dK and dV may be summed over another number of head chunks, in
    # fp32, and differ by one bf16 rounding at most, well inside 1e-2 of the norm.  dQ and,
    # for one call's chunks, dK and dV are the same bits on a second run.
    s = AttnShape(*shape)
    q, k, v, do = inputs.attn_inputs(s, seed=17)
    qd, kd, vd, o, lse = gpu_fwd(q, k, v, s.n, mode)
    dod = do.cuda()
    ws = guards.empty((binding.sfa_bwd_workspace_bytes(s.B, s.L, s.n, s.Hq, s.Hkv, s.Dh, mode),), torch.uint8)
    outs = []
    for phased in (False, True, False):
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        dq, dk, dv = guards.like(qd), guards.like(kd), guards.like(vd)
        if phased:
            binding.sfa_bwd_prep(o, dod, lse, s.n, mode, ws, s.Hkv)
            binding.sfa_bwd_main(qd, kd, vd, dod, dk, dv, s.n, mode, ws, dev_status=st)
            binding.sfa_bwd_finalize(dq, s.n, mode, ws, s.Hkv)
        else:
            binding.sfa_bwd(qd, kd, vd, o, lse, dod, dq, dk, dv, s.n, mode, ws, dev_status=st)
        check_status(st)
        outs.append([x.cpu() for x in (dq, dk, dv)])
    assert torch.equal(outs[0][0].view(torch.int16), outs[1][0].view(torch.int16))
    assert_grads_close(list(zip(("dk", "dv"), outs[1][1:], outs[0][1:])))
    for a, b in zip(outs[0], outs[2]):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
