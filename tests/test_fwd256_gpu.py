"""The head-dim-256 forward's pairs of 128-row query tiles at their edges: two heads of one
K/V group (even groups) and two tiles of one head (odd groups, whose second tile may be
empty or run one key tile longer), the K/V ring around its wrap (ten pieces, four per key
tile), and the rescaling of O, which both threads of a row carry out (Eq. 4, Fig. 2)."""
import pytest
import torch

import oracle
from paper_2607_08186_gb300 import build, inputs
from paper_2607_08186_gb300.inputs import AttnShape, CROSS, LOCAL, WITHIN

from parity import assert_fwd_close, check_status, gpu_fwd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _check(q, k, v, n, mode, window=0):
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    _, _, _, o, lse = gpu_fwd(q, k, v, n, mode, 0.0, window, status=st)
    check_status(st)
    o_ref, lse_ref = oracle.sfa_fwd(q, k, v, n, mode, None, window)
    assert_fwd_close(o.cpu(), lse.cpu(), o_ref, lse_ref)


@pytest.mark.parametrize("rows", [1, 127, 128, 129, 255, 256, 257, 385, 513, 641, 900])
@pytest.mark.parametrize("Hq,Hkv", [(2, 2), (2, 1), (3, 1)])
def test_pair_edges(rows, Hq, Hkv):
    for B, n, mode, window in ((1, 1, CROSS, 0), (2, 2, WITHIN, 0), (1, 1, LOCAL, 130), (1, 1, LOCAL, 20)):
        q, k, v = inputs.attn_inputs(AttnShape(B, rows, n, Hq, Hkv, 256), seed=rows + 7 * Hq, with_grad=False)
        _check(q, k, v, n, mode, window)


@pytest.mark.parametrize("Hq", [2, 3])
def test_rescale_per_tile(Hq):
    # keys that grow along the sequence: in the rows with positive scores the running maximum
    # grows by far more than 2^8 from one key tile to the next, in the others never
    q, k, v = inputs.attn_inputs(AttnShape(1, 600, 1, Hq, 1, 256), seed=5, with_grad=False)
    k = (k.float() * torch.linspace(0.1, 24, 600)[None, :, None, None]).to(torch.bfloat16)
    _check(q, k, v, 1, CROSS)
