"""Kernel variants and launch shapes that are chosen by size: each at the edges
of the sizes that choose it, against the oracle or a plain copy."""
import importlib

import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mw():
    return importlib.import_module("paper_2608_01127_gb300")


@pytest.mark.parametrize("H", [1, 2, 3, 4, 5, 6, 7, 11, 13])  # heads in flight: 1 to 6
@pytest.mark.parametrize("d,N", [(64, 33), (72, 28), (72, 29), (80, 26), (88, 22), (96, 43),
                                 (104, 20), (112, 17), (120, 35), (128, 31)])
def test_qkv_split_token_blocks(mw, H, d, N):
    """A block of tokens fills the threads once (twice at d = 128): at, below
    and above a block's size; V and unrotated channels bit for bit, rotated
    ones as the oracle rounds them (one bf16 ulp, plus what the 1e-6 rad of the
    angle leaves where the two products cancel)."""
    g = torch.Generator().manual_seed(d * 100 + N + H)
    qkv = torch.randn(2, N, 3, H, d, generator=g).to(torch.bfloat16)
    rope = d // 2 // 2 * 2 - 2  # ends inside a 16-byte piece for most d
    q, k, v = mw.mw_qkv_rope_split(qkv.cuda(), rope, 1e4, 9, 5)
    ref = oracle.qkv_split_rope(qkv, rope, 1e4, 9, 5)
    assert torch.equal(v.cpu(), qkv[:, :, 2].permute(0, 2, 1, 3))
    for got, want in ((q, ref[0]), (k, ref[1])):
        got = got.cpu().double()
        assert torch.equal(got[..., rope:], want[..., rope:].double())
        err = (got - want).abs()
        assert bool((err <= want.abs() * 2.0 ** -7 + 2.0 ** -16).all())


@pytest.mark.parametrize("d", [64, 72, 80, 96, 120, 128])
def test_output_rows_at_16_and_32_bytes(mw, d):
    """O, dK and dV rows go out as 32-byte stores where every row starts at a
    multiple of 32 bytes, else as 16-byte ones: the same bits either way, and
    nothing written beyond the outputs."""
    B, H, N, T = 1, 2, 150, 50
    g = torch.Generator("cuda").manual_seed(d)
    q, k, v, do = (torch.randn(B, H, N, d, generator=g, device="cuda").to(torch.bfloat16)
                   for _ in range(4))
    n = B * H * N * d
    results = []
    for shift in (16, 8):  # in elements: 32 and 16 bytes
        bufs = [torch.full((n + 64,), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(4)]
        o, dq, dk, dv = (b[shift:shift + n].view(B, H, N, d) for b in bufs)
        _, lse = mw.mw_bca_fwd(q, k, v, T, out=(o, torch.empty(B, H, N, device="cuda")))
        mw.mw_bca_bwd(q, k, v, o, lse, do, T, out=(dq, dk, dv))
        for b in bufs:
            assert bool((b[:shift] == 7).all()) and bool((b[shift + n:] == 7).all())
        results.append((o, dk, dv, lse))
    for a, b in zip(*results):
        assert torch.equal(a, b)
    o_ref, _ = oracle.fwd(q.cpu(), k.cpu(), v.cpu(), T, d ** -0.5)
    assert float((results[0][0].double().cpu() - o_ref).norm() / o_ref.norm()) <= 5e-3


@pytest.mark.parametrize("rise", [8.0, 0.0, -8.0])  # of the scores, from a 128-key tile to the next
@pytest.mark.parametrize("d", [64, 72, 80])
@pytest.mark.parametrize("T,n", [(1, 1), (64, 1), (128, 1), (129, 1), (257, 1), (100, 5), (300, 3)])
def test_weights_in_columns_of_their_own(mw, T, n, d, rise):
    """Up to 80 channels a tile's weights are split over two column ranges and
    begun with the maximum of the tiles before it: maxima that grow by more
    than 2^8 in each tile (all weights redone, O rescaled), that hardly move,
    and that fall, over one to eight key tiles.  The weights and O are rounded
    to bf16 (2^-9 each): 5e-3 of O's norm, 2^-8 of the row sum."""
    g = torch.Generator().manual_seed(d * 1000 + T * 7 + n)
    N = n * T
    q, k, v = (torch.randn(1, 3, N, d, generator=g).to(torch.bfloat16) for _ in range(3))
    q[..., 0] = d ** 0.5
    k[..., 0] = rise * (torch.arange(N) // 128)
    o, lse = mw.mw_bca_fwd(q.cuda(), k.cuda(), v.cuda(), T)
    o_ref, lse_ref = oracle.fwd(q, k, v, T, d ** -0.5)
    assert float((o.cpu().double() - o_ref).norm() / o_ref.norm()) <= 5e-3
    assert float((lse.cpu().double() - lse_ref).abs().max()) <= 2.0 ** -8


@pytest.mark.parametrize("d,rope", [(64, 64), (64, 6), (72, 24), (80, 80), (128, 32)])
@pytest.mark.parametrize("W,T,length,sink", [(1, 64, 0, 32), (1, 128, 300, 130), (2, 100, 640, 300), (3, 200, 512, 16)])
def test_turned_sink_without_a_split(mw, W, T, length, sink, d, rope):
    """The sink's key tiles turned by one helper warp (d = 64: its sibling
    issues MMAs) or by two, key range in one piece, one query tile or more:
    the tolerances of the split form's parity."""
    g = torch.Generator().manual_seed(d * 10 + W + sink)
    cap, head, shift, sc = 640, 100, 12, d ** -0.5
    q, kn, vn = (torch.randn(1, 2, W * T, d, generator=g).to(torch.bfloat16) for _ in range(3))
    kr, vr = (torch.randn(1, 2, cap, d, generator=g).to(torch.bfloat16) for _ in range(2))
    ks, vs = (torch.randn(1, 2, sink, d, generator=g).to(torch.bfloat16) for _ in range(2))
    mw.mw_set_option("cache_splits", 1)
    try:
        o, lse = mw.mw_bca_cache_fwd_rope(q.cuda(), kn.cuda(), vn.cuda(), ks.cuda(), vs.cuda(), kr.cuda(),
                                          vr.cuda(), head, length, T, rope, 1e4, shift, sc)
    finally:
        mw.mw_set_option("cache_splits", 0)
    o_ref, lse_ref = oracle.cache_fwd_reshift(q, kn, vn, kr, vr, cap, head, length, T, sc, ks, vs, rope, 1e4, shift)
    o, lse = o.cpu().double(), lse.cpu().double()
    assert float((o - o_ref).norm() / o_ref.norm()) <= 5e-3 and float((o - o_ref).abs().max()) <= 2e-2
    assert bool(((lse - lse_ref).abs() <= 1e-3 * lse_ref.abs().clamp(min=1)).all())
