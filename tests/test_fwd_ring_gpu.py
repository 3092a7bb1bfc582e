"""The forward's K/V ring at its wrap-arounds (five tiles at head dim 128, ten at 64): key
tile counts on both sides of a lap, with a CTA's two query tiles from two heads (even
groups) and from one head (odd groups, whose second tile runs one key tile longer), causal
and windowed (Eq. 4, Fig. 2)."""
import pytest
import torch

import oracle
from paper_2607_08186_gb300 import build, inputs
from paper_2607_08186_gb300.inputs import AttnShape, CROSS, LOCAL

from parity import assert_fwd_close, check_status, gpu_fwd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("Dh", [64, 128])
@pytest.mark.parametrize("Hq", [2, 3])
@pytest.mark.parametrize("rows", [127, 129, 257, 385, 513, 641, 769, 1281])
def test_ring_laps(rows, Hq, Dh):
    s = AttnShape(1, rows, 1, Hq, 1, Dh)
    q, k, v = inputs.attn_inputs(s, seed=rows + Hq, with_grad=False)
    for mode, window in ((CROSS, 0), (LOCAL, 300)):
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        _, _, _, o, lse = gpu_fwd(q, k, v, s.n, mode, 0.0, window, status=st)
        check_status(st)
        o_ref, lse_ref = oracle.sfa_fwd(q, k, v, s.n, mode, None, window)
        assert_fwd_close(o.cpu(), lse.cpu(), o_ref, lse_ref)
