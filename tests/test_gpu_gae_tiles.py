"""aht_gae at the edges of its blocks of 32 envs, warps of 4 steps and tiles of 64, against a
plain fp64 reverse scan; and with the targets written over the values."""
import pytest
import torch

from gpu_util import require_gpu
from paper_2609_13716_gb300 import aht

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 32, 33, 1000])
@pytest.mark.parametrize("T", [1, 3, 4, 5, 63, 64, 65, 128, 200])
def test_matches_a_reverse_scan(n, T):
    require_gpu()
    g = torch.Generator().manual_seed(1000 * T + n)
    r = torch.randn(T, n, generator=g)
    v = torch.randn(T, n, generator=g)
    d = (torch.rand(T, n, generator=g) < 0.1).to(torch.uint8)
    last = torch.randn(n, generator=g)
    want = torch.empty(T, n, dtype=torch.float64)
    a, nv = torch.zeros(n, dtype=torch.float64), last.double()
    for t in reversed(range(T)):
        live = 1.0 - d[t].double()
        a = r[t].double() + 0.99 * live * nv - v[t].double() + 0.99 * 0.95 * live * a
        want[t], nv = a, v[t].double()
    values = v.cuda()
    adv, tgt = torch.empty(T, n, device="cuda"), torch.empty(T, n, device="cuda")
    aht.aht_gae(r.cuda(), values, d.cuda(), last.cuda(), 0.99, 0.95, adv, tgt)
    # a sum of at most T terms that decay by 0.94, each of fp32 rounding: ~20 x 2^-24 x |A|
    torch.testing.assert_close(adv.cpu().double(), want, rtol=1e-5, atol=1e-5)
    torch.testing.assert_close(tgt.cpu().double(), want + v.double(), rtol=1e-5, atol=1e-5)
    again = torch.empty_like(adv)
    aht.aht_gae(r.cuda(), values, d.cuda(), last.cuda(), 0.99, 0.95, again, values)
    assert torch.equal(again, adv) and torch.equal(values, tgt)
