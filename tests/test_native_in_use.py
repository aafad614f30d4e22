"""The native half of the Python binding is there and takes the common calls: a
build or a check that silently sends every call the longer way is a failure."""
import importlib
import shutil

import pytest
import torch


@pytest.fixture()
def mw():
    from paper_2608_01127_gb300 import _build
    _build.build()
    m = importlib.import_module("paper_2608_01127_gb300")
    m.library()
    return m


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_it_is_built_and_loaded(mw):
    assert mw._native is not None


def test_its_absence_is_told(mw, monkeypatch, tmp_path):
    monkeypatch.setattr(mw, "_native", None)
    monkeypatch.setattr(mw, "_native_path", str(tmp_path / "_mw_torch.so"))
    with pytest.warns(RuntimeWarning, match="is missing"):
        mw._load_native(mw.library())
    (tmp_path / "_mw_torch.so").write_bytes(b"not a module")
    with pytest.warns(RuntimeWarning, match="was not loaded"):
        mw._load_native(mw.library())
    assert mw._native is None


class Spy:
    """Counts the calls that the native module answers."""

    def __init__(self, module):
        self.module, self.taken, self.left = module, [], []

    def __getattr__(self, name):
        def call(*args):
            r = getattr(self.module, name)(*args)
            (self.left if r is None else self.taken).append(name)
            return r
        return call


@pytest.mark.gpu
def test_common_calls_are_taken(mw, monkeypatch):
    def bf(*shape):
        return torch.randn(*shape, device="cuda").to(torch.bfloat16)

    spy = Spy(mw._native)
    monkeypatch.setattr(mw, "_native", spy)
    q, k, v, do = (bf(1, 2, 128, 64) for _ in range(4))
    kc, vc = bf(1, 2, 512, 64), bf(1, 2, 512, 64)
    ks, vs = bf(1, 2, 40, 64), bf(1, 2, 40, 64)
    o, lse = mw.mw_bca_fwd(q, k, v, 64)
    mw.mw_bca_fwd(q, k, v, 32, 0.2, need_lse=False)
    mw.mw_bca_bwd(q, k, v, o, lse, do, 64)
    mw.mw_bca_cache_fwd(q, k, v, kc, vc, 0, 512, 64, workspace=torch.empty(1 << 22, dtype=torch.uint8, device="cuda"))
    mw.mw_bca_cache_fwd_sink(q, k, v, ks, vs, kc, vc, 9, 300, 64)
    mw.mw_bca_cache_fwd_rope(q, k, v, ks, vs, kc, vc, 9, 300, 64, 32, 10000.0, 7)
    mw.mw_bca_cache_step(q, k, v, kc, vc, 400, 300, 188, 64, 64)
    mw.mw_qkv_rope_split(bf(1, 100, 3, 2, 72), 30, 10000.0, 7, 3)
    x = [t.clone().requires_grad_() for t in (q, k, v)]
    mw.BlockCausalAttention.apply(*x, 64, None).backward(do)
    with torch.inference_mode():
        mw.mw_bca_fwd(q, k, v, 64)
    torch.cuda.synchronize()
    assert spy.left == []
    assert spy.taken == ["fwd", "fwd", "bwd", "cache", "cache", "cache", "cache", "qkv", "fwd", "bwd", "fwd"]
