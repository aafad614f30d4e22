"""The native half of the Python binding (csrc/mw_torch.cpp) against the
binding's own checks: it takes only arguments that need nothing special, gives
bit for bit the same results, and leaves every refusal to those checks."""
import importlib

import pytest
import torch


@pytest.fixture()
def mw():
    m = importlib.import_module("paper_2608_01127_gb300")
    m.library()
    if m._native is None:
        pytest.skip("csrc/mw_torch.cpp was not built")
    return m


def test_takes_nothing_unusual(mw):
    q = torch.zeros(1, 2, 64, 64, dtype=torch.bfloat16)  # not on a GPU
    n = mw._native
    assert n.fwd(q, q, q, 64, None, True) is None
    assert n.fwd(q, q, None, 64, None, True) is None
    assert n.fwd(1, 2, 3, 4, 5, 6) is None
    assert n.fwd(q) is None
    assert n.bwd(q, q, q, q, q, q, 64, None) is None
    assert n.cache(q, q, q, None, None, q, q, 0, 64, 64, None, True, None, None, None) is None
    assert n.qkv(q, 0, 10000.0, 1, 0) is None


CASES = ["fwd", "fwd_no_lse", "bwd", "cache", "cache_ws", "sink", "rope", "step", "qkv"]


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES)
def test_same_bits_as_the_checked_way(mw, case, monkeypatch):
    g = torch.Generator("cuda").manual_seed(5)

    def bf(*shape):
        return torch.randn(*shape, generator=g, device="cuda").to(torch.bfloat16)

    # one query tile against one key tile a head: the backward's dQ has one
    # summand, so its bits do not depend on the order of the additions
    q, k, v, do = (bf(1, 3, 128, 64) for _ in range(4))
    ring = [bf(1, 3, 512, 64) for _ in range(2)]
    sink = [bf(1, 3, 40, 64) for _ in range(2)]
    qkv = bf(1, 100, 3, 2, 72)
    o, lse = mw.mw_bca_fwd(q, k, v, 64)
    ws = torch.empty(1 << 22, dtype=torch.uint8, device="cuda")

    def run():
        kc, vc = (t.clone() for t in ring)
        if case == "fwd":
            return mw.mw_bca_fwd(q, k, v, 64)
        if case == "fwd_no_lse":
            return mw.mw_bca_fwd(q, k, v, 32, 0.2, need_lse=False)
        if case == "bwd":
            return mw.mw_bca_bwd(q, k, v, o, lse, do, 64)
        if case == "cache":
            return mw.mw_bca_cache_fwd(q, k, v, kc, vc, 400, 300, 64)
        if case == "cache_ws":
            return mw.mw_bca_cache_fwd(q, k, v, kc, vc, 0, 512, 128, 0.1, workspace=ws)
        if case == "sink":
            return mw.mw_bca_cache_fwd_sink(q, k, v, *sink, kc, vc, 9, 300, 64, need_lse=False)
        if case == "rope":
            return mw.mw_bca_cache_fwd_rope(q, k, v, *sink, kc, vc, 9, 300, 64, 32, 10000.0, 7)
        if case == "step":
            return (*mw.mw_bca_cache_step(q, k, v, kc, vc, 400, 300, 188, 64, 64), kc, vc)
        return mw.mw_qkv_rope_split(qkv, 30, 10000.0, 7, 3)

    native = run()
    monkeypatch.setattr(mw, "_native", None)
    checked = run()
    assert len(native) == len(checked)
    for a, b in zip(native, checked):
        assert (a is None) == (b is None)
        assert a is None or (a.dtype == b.dtype and torch.equal(a, b))


@pytest.mark.gpu
def test_refusals_are_the_checked_ones(mw):
    q = torch.zeros(1, 2, 64, 64, dtype=torch.bfloat16, device="cuda")
    ring = torch.zeros(2, 1, 2, 256, 64, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(ValueError, match="T_chunk must be >= 1"):
        mw.mw_bca_fwd(q, q, q, 0)
    with pytest.raises(ValueError, match="not a multiple"):
        mw.mw_bca_fwd(q, q, q, 48)
    with pytest.raises(TypeError):
        mw.mw_bca_fwd(q, q.float(), q, 64)
    with pytest.raises(ValueError, match="contiguous"):
        mw.mw_bca_fwd(q.transpose(2, 3), q, q, 64)
    with pytest.raises(ValueError, match="on cpu"):
        mw.mw_bca_fwd(q, q.cpu(), q, 64)
    with pytest.raises(mw.MWError, match="scale must be > 0"):
        mw.mw_bca_fwd(q, q, q, 64, -1.0)
    with pytest.raises(ValueError, match="overlaps"):
        mw.mw_bca_cache_step(q, q, q, ring[0], ring[0], 0, 64, 64, 64, 64)
    # a workspace of the ring's bytes, large enough to be used
    need = mw.mw_bca_cache_workspace_size(1, 2, 1, 64, 64, 64)
    both = torch.zeros(2, 1, 2, max(256, need), 64, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(ValueError, match="overlaps"):
        mw.mw_bca_cache_fwd(q, q, q, both[0], both[1], 0, 64, 64,
                            workspace=both[0].reshape(-1).view(torch.uint8))
