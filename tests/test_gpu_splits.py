"""The combine of split key ranges, one kernel variant for each of 2 to 8 splits
and one for more (eight at a time): each count, with splits that hold keys and
splits that hold none, at row counts around a block's, with the commit that
shares its launch."""
import importlib

import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mw():
    return importlib.import_module("paper_2608_01127_gb300")


@pytest.mark.parametrize("splits", list(range(2, 17)))
@pytest.mark.parametrize("d,T,length", [(64, 32, 2050), (64, 33, 140), (72, 1, 2050), (120, 16, 1200),
                                        (128, 17, 300), (128, 130, 2050)])
def test_every_split_count(mw, splits, d, T, length):
    """The tolerances of the cache forward's parity (5e-3 of O's norm, 2e-2 of an
    element, 1e-3 of the LSE); ring rows bit for bit."""
    g = torch.Generator().manual_seed(d * 1000 + T * 16 + splits)
    cap, head, rows, sc = 2100, 1999, min(T, 20), d ** -0.5
    slot = (head + length) % cap
    q, kn, vn = (torch.randn(1, 3, T, d, generator=g).to(torch.bfloat16) for _ in range(3))
    kr, vr = (torch.randn(1, 3, cap, d, generator=g).to(torch.bfloat16) for _ in range(2))
    kc, vc = kr.cuda(), vr.cuda()
    mw.mw_set_option("cache_splits", splits)
    try:
        o, lse = mw.mw_bca_cache_step(q.cuda(), kn.cuda(), vn.cuda(), kc, vc, head, length, slot, rows, T, sc)
    finally:
        mw.mw_set_option("cache_splits", 0)
    o_ref, lse_ref = oracle.cache_fwd(q, kn, vn, kr, vr, cap, head, length, T, sc)
    o, lse = o.cpu().double(), lse.cpu().double()
    assert float((o - o_ref).norm() / o_ref.norm()) <= 5e-3 and float((o - o_ref).abs().max()) <= 2e-2
    assert bool(((lse - lse_ref).abs() <= 1e-3 * lse_ref.abs().clamp(min=1)).all())
    at = (slot + torch.arange(rows)) % cap
    for ring, before, new in ((kc, kr, kn), (vc, vr, vn)):
        before[:, :, at] = new[:, :, :rows]
        assert torch.equal(ring.cpu(), before)
