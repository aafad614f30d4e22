"""The native half of the Python binding is only used when it was built for the
PyTorch and Python that are running."""
import importlib
import sys
import warnings

import pytest
import torch


@pytest.fixture()
def mw(monkeypatch):
    from paper_2608_01127_gb300 import _build
    _build.build()
    m = importlib.import_module("paper_2608_01127_gb300")
    m.library()
    monkeypatch.setattr(m, "_native", None)
    return m


def test_loads_where_it_was_built(mw):
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        mw._load_native(mw.library())
    assert mw._native is not None


@pytest.mark.parametrize("version", ["2.0.0", str(torch.__version__).split("+")[0], torch.__version__ + "x"])
def test_another_pytorch_is_refused(mw, monkeypatch, version):
    if version == torch.__version__:
        pytest.skip("a PyTorch without a local version")
    monkeypatch.setattr(torch, "__version__", version)
    with pytest.warns(RuntimeWarning, match="PyTorch"):
        mw._load_native(mw.library())
    assert mw._native is None


def test_another_python_is_refused(mw, monkeypatch):
    monkeypatch.setattr(sys, "hexversion", sys.hexversion + 0x10000)
    with pytest.warns(RuntimeWarning, match="Python"):
        mw._load_native(mw.library())
    assert mw._native is None
