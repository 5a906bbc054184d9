"""The module that marshals the per-step calls belongs to one interpreter's ABI."""
import importlib.machinery
import os
import sysconfig


def test_native_module_is_named_for_its_interpreter():
    from paper_2511_13587_b200 import build
    build.build()
    from paper_2511_13587_b200 import binding
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert "cpython" in suffix and suffix in importlib.machinery.EXTENSION_SUFFIXES
    assert os.path.basename(build.NATIVE) == "_native" + suffix
    assert os.path.samefile(binding._native.__file__, build.NATIVE)
    assert not os.path.exists(os.path.join(build.PKG, "_native.so"))      # what every version would load


def test_an_untagged_module_of_an_earlier_build_goes(tmp_path, monkeypatch):
    from paper_2511_13587_b200 import build
    stale = tmp_path / "_native.so"
    stale.write_bytes(b"of another version")
    monkeypatch.setattr(build, "NATIVE_UNTAGGED", str(stale))
    build.build()
    assert not stale.exists()
