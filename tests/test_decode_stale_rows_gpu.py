"""Decoding from a cache whose rows past each sequence were never written (an allocation without
initialisation may hold infinities and NaN there): a step reads nothing from them, so it gives
the bits of the same step on a cache that holds zeros there.  Lengths whose last key tile is
full, nearly full and of one token, at every head dim and on both kernels of head dim 256."""
import pytest
import torch

import guards
from paper_2607_08186_gb300 import binding, build, inputs
from paper_2607_08186_gb300.inputs import CROSS, LOCAL, WITHIN

from parity import check_status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("mode,window", [(WITHIN, 0), (CROSS, 0), (LOCAL, 100)])
@pytest.mark.parametrize("n,Hq,Hkv,Dh", [(2, 4, 2, 64), (4, 32, 8, 128), (4, 24, 2, 256), (3, 6, 2, 256), (8, 64, 2, 256)])
def test_rows_past_the_sequence(n, Hq, Hkv, Dh, mode, window):
    Lcap = 300
    lens = torch.tensor([1, 16, 31, 32, 33, 64, 65, 171, Lcap - 1, Lcap], dtype=torch.int32)
    B = len(lens)
    q = inputs.normal_bf16((B, n, Hq, Dh), Dh + n).cuda()
    kc = inputs.normal_bf16((B, Lcap * n, Hkv, Dh), Dh + n + 1).cuda()
    vc = inputs.normal_bf16((B, Lcap * n, Hkv, Dh), Dh + n + 2).cuda()
    ld = lens.cuda()
    stale = torch.arange(Lcap * n, device="cuda")[None, :] >= (ld * n)[:, None]
    ws = guards.empty((binding.sfa_decode_workspace_bytes(B, Lcap, n, Hq, Hkv, Dh, mode, window),), torch.uint8)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = None
    for fill in (0.0, float("nan"), float("inf"), float("-inf")):
        kc[stale], vc[stale] = fill, fill
        o = guards.like(q)
        lse = guards.empty((B, Hq, n), torch.float32)
        binding.sfa_decode(q, kc, vc, ld, o, n, mode, ws, lse=lse, window=window, dev_status=st)
        check_status(st)
        got = o.view(torch.int16).cpu(), lse.view(torch.int32).cpu()
        if ref is None:
            ref = got
            assert torch.isfinite(o).all() and torch.isfinite(lse).all()
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]), fill
