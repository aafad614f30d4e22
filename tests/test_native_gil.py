"""The native half of the Python binding and the interpreter lock: an exception
out of the part of a call that runs without the lock reaches Python."""
import os
import subprocess
import sys
import textwrap

import pytest

from paper_2608_01127_gb300 import _build

PROBE = r"""
#include "mw_torch.cpp"
#include <stdexcept>
namespace {
PyObject* throws(PyObject*, PyObject*) {
  HANDLE_TH_ERRORS
  call([]() -> mw_status { throw std::runtime_error("thrown without the lock"); });
  return none();
  END_HANDLE_TH_ERRORS
}
PyMethodDef probe_methods[] = {{"throws", throws, METH_NOARGS, ""}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef probe = {PyModuleDef_HEAD_INIT, "_probe", nullptr, -1, probe_methods,
                     nullptr, nullptr, nullptr, nullptr};
}  // namespace
PyMODINIT_FUNC PyInit__probe(void) { return PyModule_Create(&probe); }
"""


@pytest.mark.slow
def test_an_exception_without_the_lock_reaches_python(tmp_path):
    source, module = tmp_path / "probe.cpp", tmp_path / "_probe.so"
    source.write_text(PROBE)
    command = _build._torch_module()
    command[command.index(os.path.join(_build.CSRC, _build.TORCH_SOURCE))] = str(source)
    command[command.index("-o") + 1] = str(module)
    subprocess.run([*command, "-I" + _build.CSRC], check=True, capture_output=True)
    code = f"""
        import importlib.util, torch
        spec = importlib.util.spec_from_file_location("_probe", {str(module)!r})
        m = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(m)
        for _ in range(3):
            try:
                m.throws()
            except RuntimeError as e:
                print("raised", e)
    """
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.count("raised thrown without the lock") == 3
