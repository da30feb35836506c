"""The build's Python module (no GPU needed)."""
import sys
import sysconfig

import pytest

import paper_2607_10582_gb300 as md
from paper_2607_10582_gb300 import build as mdbuild


def test_binding_is_named_for_the_interpreter_that_built_it():
    """Another Python version neither loads the file nor takes it for its own
    build."""
    assert mdbuild.BINDING_PATH.endswith("_calls" + sysconfig.get_config_var("EXT_SUFFIX"))


def test_library_builds_and_binds_without_python_headers(monkeypatch, tmp_path):
    """Where Python.h is missing the C module is left out and the per-step calls
    go through ctypes; where it is there, a missing module is an error."""
    monkeypatch.setattr(mdbuild, "BINDING_PATH", str(tmp_path / "_calls.so"))
    monkeypatch.setattr(md, "_fast", None)
    monkeypatch.delattr(md, "_calls", raising=False)
    monkeypatch.setitem(sys.modules, md.__name__ + "._calls", None)      # the import fails
    with pytest.raises(RuntimeError, match="missing"):
        md._binding()
    monkeypatch.setattr(mdbuild.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    mdbuild.build()
    assert not (tmp_path / "_calls.so").exists()
    b = md._binding()
    assert b.decode_step(None, 1, None, None, None, b"", None) is None
    c = object.__new__(md.Cache)
    c.h = c._hv = None
    c._b, c.max_batch, c.torch, c.device = b, 4, pytest.importorskip("torch"), "cpu"
    c._specs = {md.MD_STATE_A: ((4,), c.torch.float32)}
    for call in (lambda: c.decode_step(1, None, None, None, [6], None),
                 lambda: c.decode_layer(0, 1, None, None, None, [6], None),
                 lambda: c.evict(md.np.array([1], "int32")), lambda: c.get_state(md.MD_STATE_A)):
        with pytest.raises(md.MemDecayError, match="null handle"):
            call()
