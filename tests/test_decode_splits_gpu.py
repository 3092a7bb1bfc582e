"""The decoding step's splits (Sec. 3.2): each sequence's own range over all of them, so short
sequences beside a long one leave some empty; more partials than the combine pass holds in
flight at once (67 and 71 splits); streams whose count does not divide a 32-column word (the
head-dim-256 stream masks), and windows; against the oracle."""
import pytest
import torch

from paper_2607_08186_gb300 import inputs

from test_decode_gpu import CROSS, LOCAL, WITHIN, _built, _case, _check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lcap,Dh", [(9000, 64), (9000, 128), (17000, 256)])
def test_many_splits(Lcap, Dh):
    q, kc, vc = _case(1, Lcap, 1, 4, 1, Dh, 5)
    for T in (Lcap, 130):
        _check(q, kc, vc, torch.tensor([T], dtype=torch.int32), 1, CROSS)


@pytest.mark.parametrize("n,Hq,Hkv", [(1, 24, 2), (3, 12, 2), (5, 6, 1), (8, 8, 1), (32, 4, 1), (33, 3, 1)])
@pytest.mark.parametrize("mode,w", [(WITHIN, 0), (CROSS, 0), (LOCAL, 150)])
def test_head_dim_256_streams(n, Hq, Hkv, mode, w):
    Lcap = 400 // n + 70
    q, kc, vc = _case(4, Lcap, n, Hq, Hkv, 256, n + Hq)
    _check(q, kc, vc, torch.tensor([Lcap, 1, Lcap // 2, 43], dtype=torch.int32), n, mode, w)
